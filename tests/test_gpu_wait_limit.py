"""afc_set_grid_wait_limit is a limit of the BiCGStab launches: with a limit of zero, under which
those give up, explicit steps and GMRES solves run as without it."""
import numpy as np
import pytest

from paper_2110_15676_gb300 import workloads as W
from pairs import gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_other_launches_keep_their_limit(precision):
    from paper_2110_15676_gb300 import afc
    prec = afc.AFC_MIXED if precision == "mixed" else afc.AFC_FP64
    wl = W.rotating_transient("q1", 21)
    g = gpu_problem(wl.elem, wl.n, wl.b, wl.eps, wl.c, wl.f, wl.dir_mask, wl.u_dir, family="mc", precision=precision)
    ssp = afc.default_opts(scheme=afc.AFC_SSP3, dt=g.cfl_timestep(0.5), precision=prec)
    st = afc.default_opts(limiter=afc.AFC_LIM_MC, omega=0.5, ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-2,
                          fp_fixed_its=6, precision=prec)
    rhs = np.random.default_rng(1).uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    res = []
    for limit in (4000.0, 0.0):
        g.set_grid_wait_limit(limit)
        g.set_solution(wl.u0)
        for _ in range(5):
            g.step(ssp)
        out = [g.get_solution()]
        g.solve_stationary(st)
        out.append(g.get_solution())
        out.append(g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-4, precision=prec))[0])
        res.append(out)
    for a, b in zip(*res):
        assert np.array_equal(a, b)
