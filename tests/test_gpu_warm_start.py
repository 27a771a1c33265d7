"""A stationary solve that starts from its converged solution costs one residual: the launches of the
graph form are those of the host-driven loop, and the start of the loop (its scalars and the solver
launch that stops it) beside them."""
import numpy as np
import pytest

from paper_2110_15676_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("ksp", ["gmres", "bicgstab"])
def test_converged_start_forms_one_residual(precision, ksp):
    from paper_2110_15676_gb300 import afc
    n = (9, 8, 7)
    xyz = W.grid_coords(n)
    ix, iy, iz = W.grid_index(n)
    mask = ((ix == 0) | (iy == n[1] - 1) | (iz == 0)).astype(np.uint8)
    prec = afc.AFC_MIXED if precision == "mixed" else afc.AFC_FP64
    g = afc.Problem.structured("p1", n)
    g.set_coefficients(1e-3, np.array([1.0, -0.5, 0.25]), 1.0, np.ones(len(xyz)))
    g.set_dirichlet(mask, np.where(mask, xyz[:, 1], 0.0))
    g.assemble(afc.AFC_FAMILY_MC, prec)
    o = afc.default_opts(limiter=afc.AFC_LIM_MC, omega=0.5, ksp=afc.AFC_KSP_GMRES if ksp == "gmres" else afc.AFC_KSP_BICGSTAB,
                         ksp_atol=0.0, ksp_rtol=1e-2, fp_tol=1e-8, fp_maxit=1500, precision=prec)
    g.set_solution(np.where(mask, xyz[:, 1], 0.0))
    st = g.solve_stationary(o)
    assert st["status"] == 0 and st["outer_its"] > 4
    u = g.get_solution()
    count = {}
    for graph in (0, 1):
        o.graph = graph
        g.solve_stationary(o)           # builds what the form keeps
        before = g.launches()
        st = g.solve_stationary(o)
        count[graph] = g.launches() - before
        assert st["status"] == 0 and st["outer_its"] == 0
        assert np.array_equal(g.get_solution(), u)
    assert count[1] <= count[0] + 2
