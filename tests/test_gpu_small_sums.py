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
