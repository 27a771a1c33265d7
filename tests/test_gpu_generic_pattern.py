"""Explicit and Crank-Nicolson steps on element lists whose pattern is neither structured one: the
offsets are taken three at a time, the last group reaching past the pattern by none, one or two
(39 and 45, 23 and 35, 19 offsets).  Against the oracle, and bit for bit over the launch forms."""
import numpy as np
import pytest

from oracle import afc_oracle as O

pytestmark = pytest.mark.gpu


def _l_mesh(elem, nx, ny, cut, h, nz):
    """A prism over an L in the y-z plane: ny rows of nodes in the first h layers, `cut` beyond."""
    rows = [ny if z < h else cut for z in range(nz)]
    off = np.concatenate([[0], np.cumsum(nx * np.array(rows))])
    xyz = np.concatenate([np.stack([np.tile(np.arange(nx), r), np.repeat(np.arange(r), nx), np.full(nx * r, z)], 1)
                          for z, r in enumerate(rows)]) / float(max(ny, nz) - 1)
    cells = []
    for z in range(nz - 1):
        for y in range(min(rows[z], rows[z + 1]) - 1):
            x = np.arange(nx - 1)
            v = np.stack([off[z + dz] + x + dx + nx * (y + dy) for dz in (0, 1) for dy in (0, 1) for dx in (0, 1)], 1)
            if elem == "q1":
                cells.append(v)
            else:   # Kuhn: the six paths from corner 0 to corner 7
                cells += [v[:, [0, a, b, 7]] for a, b in ((1, 3), (1, 5), (2, 3), (2, 6), (4, 5), (4, 6))]
    return xyz, np.concatenate(cells).astype(np.int32)


CASES = [("p1", (5, 7, 5, 4, 8), 23), ("p1", (3, 7, 5, 3, 6), 23), ("q1", (5, 7, 5, 4, 8), 39), ("q1", (2, 9, 5, 4, 8), 35),
         ("q1", (2, 3, 3, 2, 4), 19), ("q1", (17, 17, 9, 8, 17), 45)]


def _pair(elem, dims):
    from paper_2110_15676_gb300 import afc
    xyz, conn = _l_mesh(elem, *dims)
    N = len(xyz)
    rng = np.random.default_rng(N)
    # no entry of the convection matrix is exactly 0 (the oracle's D leaves out a pair stored on one side only)
    b = np.stack([0.5137 - xyz[:, 1], xyz[:, 0] - 0.4871, 0.1093 + 0.0 * xyz[:, 0]], 1)
    mask = (xyz[:, 1] == 0.0).astype(np.uint8)
    u = np.where(mask != 0, 0.0, rng.uniform(0.0, 1.0, N))
    g = afc.Problem.from_elements(elem, xyz, conn)
    g.set_coefficients(1e-4, b, 0.0, np.zeros(N))
    g.set_dirichlet(mask, np.zeros(N))
    g.assemble(precision=afc.AFC_MIXED)
    prob = O.assemble(O.Mesh(elem, xyz, conn.astype(np.int64)), 1e-4, b, 0.0, np.zeros(N), mask.astype(bool), np.zeros(N))
    return afc, g, prob, u


@pytest.mark.parametrize("elem,dims,K", CASES)
def test_explicit_step(elem, dims, K):
    afc, g, prob, u = _pair(elem, dims)
    assert g.info()["n_offsets"] == K
    dt = O.cfl_timestep(prob, 0.5)
    want = O.ssp_step(prob, u, dt, order=3)
    for prec in (afc.AFC_FP64, afc.AFC_MIXED):
        res = []
        for form in ("graph", "host", afc.AFC_BATCH_PER_PASS, afc.AFC_BATCH_PER_STAGE, afc.AFC_BATCH_PER_STEP):
            o = afc.default_opts(scheme=afc.AFC_SSP3, dt=dt, precision=prec)
            g.set_solution(u)
            if isinstance(form, str):
                o.graph = int(form == "graph")
                g.step(o)
            else:
                batch = afc.Batch([g])
                batch.set_tuning(form, 128)
                batch.step(o, nsteps=1)
            res.append(g.get_solution())
            assert np.array_equal(res[0], res[-1]), form
        assert np.abs(res[0] - want).max() <= (1e-12 if prec == afc.AFC_FP64 else 1e-6)


@pytest.mark.parametrize("elem,dims,K", CASES)
def test_cn_step(elem, dims, K):
    afc, g, prob, u = _pair(elem, dims)
    dt = O.cfl_timestep(prob, 1.0)
    want, _ = O.cn_step(prob, u, dt, fixed_iterations=4, ksp_atol=1e-14)
    for graph in (0, 1):
        g.set_solution(u)
        g.step(afc.default_opts(scheme=afc.AFC_CN_NONLINEAR, dt=dt, fp_fixed_its=4, ksp_atol=1e-14, graph=graph))
        assert np.abs(g.get_solution() - want).max() <= 1e-10
