"""The forms of the explicit passes: rows at which the launch changes (programmatic dependent
launch, the form for grids that do not fill the GPU) give the bits of a batch of one, whose
passes have neither; and Zalesak's sums and factors on fluxes of very different size."""
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


def _problem(afc, elem, n, precision):
    xyz = W.grid_coords(n)
    g = afc.Problem.structured(elem, n)
    g.set_coefficients(1e-6, W.rotating_b(xyz))
    g.set_dirichlet(W.boundary_mask(n), np.zeros(len(xyz)))
    g.assemble(precision=precision)
    u0 = W.front_field(xyz, np.random.default_rng(5))
    u0[W.boundary_mask(n) != 0] = 0.0
    return g, u0


# 16,384 rows and a layer more; 300,000 rows from both sides (66 x 67 x 67 = 296,274)
@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("elem,n", [("p1", (4, 3, 3)), ("q1", (16, 32, 32)), ("q1", (16, 32, 33)), ("p1", (66, 67, 67)),
                                    ("p1", (67, 67, 67)), ("q1", (67, 67, 67))])
@pytest.mark.parametrize("scheme", ["ssp2", "ssp3"])
def test_step_equals_a_batch_of_one(afc, elem, n, precision, scheme):
    prec = afc.AFC_MIXED if precision == "mixed" else afc.AFC_FP64
    g, u0 = _problem(afc, elem, n, prec)
    o = afc.default_opts(scheme=afc.AFC_SSP2 if scheme == "ssp2" else afc.AFC_SSP3, dt=g.cfl_timestep(0.5),
                         precision=prec)
    res = []
    for graph in (1, 0):
        o.graph = graph
        g.set_solution(u0)
        for _ in range(2):
            st = g.step(o)
        res.append(g.get_solution())
        assert st["umin"] == res[-1].min() and st["umax"] == res[-1].max()
    g.set_solution(u0)
    afc.Batch([g]).step(o, nsteps=2)
    res.append(g.get_solution())
    assert np.array_equal(res[0], res[1]) and np.array_equal(res[0], res[2])


@pytest.mark.parametrize("elem", ["p1", "q1"])
@pytest.mark.parametrize("decades", [3, 20, 60])
def test_factors_of_fluxes_over_decades(afc, elem, decades):
    """R+/- against the oracle on nodal values log-uniform over `decades` decades with both signs
    and zeros: the fixed-point sums shift by every amount, and small terms fall off the end.
    The sums' relative errors (2^-52 here, 25 * 2^-53 in the oracle) and the roundings of the
    predictor and the fluxes, relative to the largest neighbour, stay far below 1e-12 of a factor
    in [0, 1]: the same stage in 80-bit arithmetic is within 1e-14."""
    n = (9, 8, 7)
    xyz = W.grid_coords(n)
    N = len(xyz)
    rng = np.random.default_rng(decades)
    u = rng.choice([-1.0, 1.0], N) * 10.0 ** rng.uniform(-decades, 0.0, N)
    u[rng.uniform(size=N) < 0.1] = 0.0
    mask = W.boundary_mask(n)
    prob = O.assemble(O.structured_mesh(elem, n), 1e-6, W.rotating_b(xyz), 0.0, np.zeros(N), mask.astype(bool), np.zeros(N))
    u[mask != 0] = 0.0
    dt = O.cfl_timestep(prob, 0.5)
    g = afc.Problem.structured(elem, n)
    g.set_coefficients(1e-6, W.rotating_b(xyz))
    g.set_dirichlet(mask, np.zeros(N))
    g.assemble()
    g.set_solution(u)
    got = g.fe_stage(dt)
    want = O.fe_ssp_stage(prob, u, dt, want=True)[1]
    for k in ("Rp", "Rm"):
        assert np.max(np.abs(got[k] - want[k])) <= 1e-12, k
