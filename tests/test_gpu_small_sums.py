"""Zalesak's P+ and P- where one is far below the rounding of the other: isolated nodes of height
+-1 in a field of another scale give rows whose large fluxes all have one sign, and a factor that
the small sum of the other sign decides.  Each sum is its own: a small one is not lost beside a
large one (it would give R = 1 where R = 0)."""
import numpy as np
import pytest

from oracle import afc_oracle as O
from paper_2110_15676_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def afc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_15676_gb300 import afc as m
    return m


def _field(elem, small, sign):
    n = (12, 11, 10)
    xyz = W.grid_coords(n)
    ix, iy, iz = W.grid_index(n)
    mask = W.boundary_mask(n)
    u = small * np.random.default_rng(5).uniform(-1.0, 1.0, len(xyz))
    u[(ix % 4 == 2) & (iy % 4 == 2) & (iz % 4 == 2)] = 1.0
    u = np.where(mask != 0, 0.0, sign * u)
    b = np.tile([1.0, 0.5, 0.25], (len(xyz), 1))
    prob = O.assemble(O.structured_mesh(elem, n), 0.0, b, 0.0, np.zeros(len(xyz)), mask.astype(bool), np.zeros(len(xyz)))
    return n, b, mask, u, prob


def _problem(afc, elem, n, b, mask, u):
    g = afc.Problem.structured(elem, n)
    g.set_coefficients(0.0, b)
    g.set_dirichlet(mask, np.zeros(len(u)))
    g.assemble()
    g.set_solution(u)
    return g


def _rows(lim, ratio):
    """Rows whose P of one sign is below `ratio` of the other and decides its factor, per factor."""
    Pp, Pm = lim["Pp"], -lim["Pm"]
    return {"Rp": (Pp > 0) & (Pp < ratio * Pm) & (lim["Rp"] < 0.9), "Rm": (Pm > 0) & (Pm < ratio * Pp) & (lim["Rm"] < 0.9)}


# the last field is of subnormal fluxes (2^-1026, spaced 2^-1074: 2^-47 of a value per operation, 26
# terms, and up to 100 between the predictor's values and their difference)
@pytest.mark.parametrize("elem", ["p1", "q1"])
@pytest.mark.parametrize("small,tol", [(1e-19, 1e-12), (1e-25, 1e-12), (1e-120, 1e-12), (1e-306, 1e-9)])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_explicit_factors(afc, elem, small, tol, sign):
    n, b, mask, u, prob = _field(elem, small, sign)
    dt = 1.5 * O.cfl_timestep(prob, 1.0)
    want = O.fe_ssp_stage(prob, u, dt, want=True)[1]
    rows = _rows(want, 2.0 ** -58)
    assert rows["Rp"].any() or rows["Rm"].any()
    got = _problem(afc, elem, n, b, mask, u).fe_stage(dt)
    for k, sel in rows.items():
        assert np.all(np.abs(got[k] - want[k])[sel] <= tol), k


def _cn(prob, u, dt):
    """Fluxes, predictor and limiter of the CN residual at u_new = u_old = u."""
    ut = u - 0.5 * dt * (prob.AA @ u - prob.f) / prob.mL
    ut[prob.dir_mask] = 0.0
    return O.zalesak_limiter(prob, O.cn_fluxes(prob, u, u, dt, False), ut, dt)[1]


@pytest.mark.parametrize("elem", ["p1", "q1"])
@pytest.mark.parametrize("small", [1e-19, 1e-25])
@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_cn_factors(afc, elem, small, sign):
    n, b, mask, u, prob = _field(elem, small, sign)
    dt = 3.0 * O.cfl_timestep(prob, 1.0)
    want = _cn(prob, u, dt)
    rows = _rows(want, 2.0 ** -58)
    assert rows["Rp"].any() or rows["Rm"].any()
    got = _problem(afc, elem, n, b, mask, u).cn_limited_sum(dt, u, u, prelimit=0)
    for k, sel in rows.items():
        assert np.all(np.abs(got[k] - want[k])[sel] <= 1e-12), k


@pytest.mark.parametrize("elem", ["p1", "q1"])
def test_cn_sums_are_rounded_once(afc, elem):
    """R+/- of the CN scheme bit for bit from correctly rounded P+/- (u_new = u_old, no
    prelimiting: r_ij = d_ij (u_j - u_i), with the library's own d_ij, predictor and masses)."""
    import math
    n, b, mask, _, prob = _field(elem, 1.0, 1.0)
    N = len(mask)
    u = np.where(mask != 0, 0.0, np.random.default_rng(3).uniform(-1.0, 1.0, N))
    g = _problem(afc, elem, n, b, mask, u)
    dt = 4.0 * g.cfl_timestep(1.0)
    got = g.cn_limited_sum(dt, u, u, prelimit=0)
    rowptr, col, d = g.export_csr(afc.AFC_MAT_D)
    m, ut = g.lumped_mass(), got["u_tilde"]
    decided = 0
    for i in np.flatnonzero(mask == 0):
        at = slice(rowptr[i], rowptr[i + 1])
        j = col[at]
        r = np.where(j == i, 0.0, d[at] * (2.0 * u[j] - 2.0 * u[i])) / 2.0
        for k, P, Q in (("Rp", math.fsum(r[r > 0]), ut[j].max() - ut[i]), ("Rm", math.fsum(r[r < 0]), ut[j].min() - ut[i])):
            num, den = m[i] * Q, dt * P
            want = 1.0 if den == 0.0 or abs(num) >= abs(den) else num / den
            assert got[k][i] == want, (i, k)
            decided += want < 1.0
    assert decided > N // 4


@pytest.mark.parametrize("elem", ["p1", "q1"])
def test_explicit_factors_of_a_nan_flux(afc, elem):
    """One node is NaN.  Its neighbours' rates and predictors are NaN; a free row that is no neighbour
    of it but has one of a lower index has a finite predictor, a finite Q- (NaN sorts as a maximum) and
    a NaN flux with the sign bit set (the negative of the pair's): its P- and so its R- are NaN."""
    n, b, mask, u, prob = _field(elem, 1.0, 1.0)
    centre = np.ravel_multi_index((5, 5, 5), (n[2], n[1], n[0]))
    u[centre] = np.nan
    g = _problem(afc, elem, n, b, mask, u)
    got = g.fe_stage(0.5 * O.cfl_timestep(prob, 1.0))
    rowptr, col, _ = g.export_csr(afc.AFC_MAT_MC)
    near = [set(col[rowptr[i]:rowptr[i + 1]]) for i in range(len(mask))]
    ring = {j for j in near[centre] if mask[j] == 0}
    rows = [i for i in range(len(mask)) if mask[i] == 0 and i not in near[centre] and any(j < i for j in near[i] & ring)]
    assert len(rows) >= 20
    assert np.isfinite(got["u_tilde"][rows]).all()
    assert np.isnan(got["Rm"][rows]).all()
