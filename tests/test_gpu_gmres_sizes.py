"""GMRES(m) as one persistent launch, at the sizes where its split over blocks changes:
fewer rows than a block, one row more or less than a full grid of blocks, several rows per
thread, and rows beyond the shared memory that holds a block's share of the new direction.
The reference is the true residual of the returned solution, formed with the exported or
applied operator (no code of the solver)."""
import numpy as np
import pytest

from paper_2110_15676_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_15676_gb300 import afc as m
    return m


def _problem(afc, elem, n, precision):
    xyz = W.grid_coords(n)
    ix, iy, iz = W.grid_index(n)
    mask = ((ix == 0) | (iy == n[1] - 1) | (iz == 0)).astype(np.uint8)
    g = afc.Problem.structured(elem, n)
    g.set_coefficients(1e-3, np.array([1.0, -0.5, 0.25]), 1.0, np.ones(len(xyz)))
    g.set_dirichlet(mask, np.where(mask, xyz[:, 1], 0.0))
    g.assemble(afc.AFC_FAMILY_MC, precision)
    return g, mask


# 8 rows (one block), 63 / 64 / 65 rows, 64 * 152 = 9728 rows (one full block per SM) and one
# z-layer more, 32-row remainders, several rows per thread
SIZES = [(2, 2, 2), (7, 3, 3), (4, 4, 4), (13, 5, 1 + 1), (64, 19, 8), (64, 19, 9), (41, 33, 57), (97, 81, 65)]


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("elem", ["p1", "q1"])
@pytest.mark.parametrize("n", SIZES)
def test_gmres_true_residual(afc, elem, n, precision):
    mixed = precision == "mixed"
    g, mask = _problem(afc, elem, n, afc.AFC_MIXED if mixed else afc.AFC_FP64)
    rng = np.random.default_rng(n[0] * 100 + n[2])
    rhs = rng.uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    rtol = 1e-4 if mixed else 1e-10
    x, its, res = g.linear_solve(0, rhs, afc.default_opts(
        ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=rtol, ksp_maxit=2000,
        precision=afc.AFC_MIXED if mixed else afc.AFC_FP64))
    r = rhs - np.where(mask, x, g.apply(afc.AFC_MAT_LOW, x))
    # the solver's own true residual is below rtol |rhs|; forming it again costs a rounding of
    # the operator's rows (single precision in the mixed mode: 2^-24 relative to |A| |x|)
    slack = (2.0 ** -22 if mixed else 2.0 ** -50) * np.linalg.norm(np.where(mask, x, g.apply(afc.AFC_MAT_LOW, np.abs(x))))
    assert np.linalg.norm(r) <= 1.001 * rtol * np.linalg.norm(rhs) + 4.0 * slack
    assert abs(res - np.linalg.norm(r)) <= 0.01 * rtol * np.linalg.norm(rhs) + 4.0 * slack
    assert 0 < its < 2000


def test_gmres_rows_beyond_shared_memory(afc):
    """P1 149^3 in double precision: 21,763 rows a block, 174 KB of w: kept in global memory."""
    n = (149, 149, 149)
    g, mask = _problem(afc, "p1", n, afc.AFC_FP64)
    rhs = np.random.default_rng(7).uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    x, its, res = g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-8,
                                                          ksp_maxit=2000))
    r = rhs - np.where(mask, x, g.apply(afc.AFC_MAT_LOW, x))
    assert np.linalg.norm(r) <= 1.001e-8 * np.linalg.norm(rhs)
    assert 0 < its < 2000


@pytest.mark.parametrize("n", [(5, 5, 5), (33, 17, 25)])
def test_gmres_iteration_limit_and_zero_start(afc, n):
    """The iteration limit inside and at the end of a cycle, and a right-hand side that is
    below the tolerance at once (x = 0)."""
    g, _ = _problem(afc, "q1", n, afc.AFC_FP64)
    rhs = np.random.default_rng(3).uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    for maxit in (1, 3, 4, 5, 9):
        _, its, _ = g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-14,
                                                            ksp_maxit=maxit, gmres_restart=4))
        assert its == maxit
    x, its, res = g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_GMRES, ksp_atol=1.0, ksp_rtol=0.0))
    assert its == 0 and not x.any() and res == pytest.approx(np.linalg.norm(rhs), rel=1e-12)
