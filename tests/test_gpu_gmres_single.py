"""GMRES on single-precision vectors, bit for bit: the solution of a mixed-precision linear solve
equals that of the same iteration in numpy with every single-precision rounding in its defined
place (normalised basis; dots along strands of 256-row chunks, butterflies of 32 strands, eight
results in turn).  The scalars of both sides are doubles whose rounding may differ; one shows only
where a coefficient lies within 1e-16 of a rounding boundary of single precision, so the bits are
compared without a tolerance.  And a whole mixed stationary solve gives the same bits again."""
import math

import numpy as np
import pytest

from paper_2110_15676_gb300 import workloads as W

pytestmark = pytest.mark.gpu
F = np.float32


@pytest.fixture(scope="module")
def afc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("needs a CUDA device")
    from paper_2110_15676_gb300 import afc as m
    return m


def _problem(afc, elem, n):
    xyz = W.grid_coords(n)
    ix, iy, iz = W.grid_index(n)
    mask = ((ix == 0) | (iy == n[1] - 1) | (iz == 0)).astype(np.uint8)
    g = afc.Problem.structured(elem, n)
    g.set_coefficients(1e-3, np.array([1.0, -0.5, 0.25]), 1.0, np.ones(len(xyz)))
    g.set_dirichlet(mask, np.where(mask, xyz[:, 1], 0.0))
    g.assemble(afc.AFC_FAMILY_MC, afc.AFC_MIXED)
    return g, mask


def _fma(a, b, c):
    """a b + c rounded once to single: the exact sum rounded to odd in double, then to single."""
    p = np.asarray(a, np.float64) * b
    c = np.asarray(c, np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    even = (s.view(np.int64) & 1) == 0
    return np.where((err != 0.0) & even, np.nextafter(s, np.where(err > 0.0, np.inf, -np.inf)), s).astype(F)


def _sets(n):   # strand sets per SM of a step with n basis vectors
    return 6 if n <= 4 else 5 if n <= 12 else 4 if n <= 16 else 3 if n <= 20 else 2


class Gmres:
    def __init__(self, g, afc, mask, nsm):
        rowptr, col, val = g.export_csr(afc.AFC_MAT_LOW)
        N = self.N = len(rowptr) - 1
        row = np.repeat(np.arange(N), np.diff(rowptr))
        off = col - row
        self.offs = np.unique(off)
        self.B = np.zeros((len(self.offs), N), F)
        keep = mask[row] == 0
        self.B[np.searchsorted(self.offs, off[keep]), row[keep]] = val[keep].astype(F)
        diag = np.ones(N)
        dk = keep & (off == 0)
        diag[row[dk]] = val[dk]
        self.B[np.searchsorted(self.offs, 0), mask != 0] = F(1)
        self.dinv = (1.0 / diag).astype(F)
        self.nsm = nsm
        self.chunks = -(-N // 256)

    def product(self, z):
        pad = int(np.abs(self.offs).max())
        zp = np.zeros(self.N + 2 * pad, F)
        zp[pad:pad + self.N] = z
        y = np.zeros(self.N, F)
        for k, o in enumerate(self.offs):
            y = _fma(self.B[k], zp[pad + o:pad + o + self.N], y)
        return y

    def strands(self, w, v, n):
        G = min(_sets(n) * self.nsm, self.chunks)
        J = -(-self.chunks // G)
        wp, vp = (np.zeros(J * G * 256, F) for _ in range(2))
        wp[:self.N], vp[:self.N] = w, v
        wp, vp = wp.reshape(J, G, 256), vp.reshape(J, G, 256)
        acc = np.zeros((G, 256), F)
        for j in range(J):
            acc = _fma(wp[j], vp[j], acc)
        return acc

    def dot(self, w, v, n):
        x = self.strands(w, v, n).reshape(-1, 8, 32)
        lane = np.arange(32)
        for o in (16, 8, 4, 2, 1):
            x = x + x[:, :, lane ^ o]
        s = np.zeros(len(x), F)
        for u in range(8):
            s = s + x[:, u, 0]
        return math.fsum(s.astype(np.float64))

    def norm(self, w, n):
        return math.sqrt(math.fsum(self.strands(w, w, n).astype(np.float64).ravel()))

    def solve(self, rhs, m, rtol, maxit):
        x = np.zeros(self.N, F)
        its, first, tol = 0, True, None
        while True:
            w = rhs.astype(F) - (F(0) if first else self.product(x))
            beta = math.sqrt(math.fsum((w * w).astype(np.float64)))
            if first:
                tol = rtol * beta
            first = False
            if beta < tol or its >= maxit:
                return x, its
            V = [w * F(1.0 / beta)]
            H = np.zeros((m + 1, m))
            g, cs, sn = np.zeros(m + 1), np.zeros(m), np.zeros(m)
            g[0] = beta
            for k in range(m):
                w = self.product(self.dinv * V[k])
                h = np.array([self.dot(w, v, k + 1) for v in V])
                ww = self.dot(w, w, k + 1)
                H[:k + 1, k] = h
                for q in range(k + 1):
                    w = _fma(-F(h[q]), V[q], w)
                if not ww - (h * h).sum() >= 0.5 * ww:
                    h = np.array([self.dot(w, v, k + 1) for v in V])
                    H[:k + 1, k] += h
                    for q in range(k + 1):
                        w = _fma(-F(h[q]), V[q], w)
                hk1 = self.norm(w, k + 1)
                for q in range(k):
                    a, b = H[q, k], H[q + 1, k]
                    H[q, k], H[q + 1, k] = cs[q] * a + sn[q] * b, -sn[q] * a + cs[q] * b
                den = math.hypot(H[k, k], hk1)
                cs[k], sn[k] = H[k, k] / den, hk1 / den
                H[k, k] = den
                g[k + 1], g[k] = -sn[k] * g[k], cs[k] * g[k]
                its += 1
                V.append(w * F(1.0 / hk1))
                if abs(g[k + 1]) < tol or its >= maxit:
                    break
            ku = k + 1
            y = np.zeros(ku)
            for q in range(ku - 1, -1, -1):
                y[q] = (g[q] - H[q, q + 1:ku] @ y[q + 1:ku]) / H[q, q]
            s = np.zeros(self.N, F)
            for q in range(ku):
                s = _fma(F(y[q]), V[q], s)
            x = _fma(self.dinv, s, x)


# less than a chunk; whole chunks (512 rows) and a remainder; the last size of one or two chunks a
# block (302 chunks on 151 blocks) and beyond it, with more than 20 vectors (strands of two rows);
# strands of two rows from the first vector on, with the basis in shared memory and past it
CASES = [("p1", (5, 4, 3), 20, 9), ("q1", (16, 16, 2), 4, 9), ("p1", (13, 11, 7), 32, 26), ("p1", (41, 33, 57), 9, 12),
         ("q1", (52, 43, 44), 32, 24), ("p1", (64, 64, 64), 6, 8), ("q1", (65, 65, 65), 6, 8), ("p1", (97, 65, 71), 17, 18)]


@pytest.mark.parametrize("elem,n,m,maxit", CASES)
def test_solution_bits(afc, elem, n, m, maxit):
    import torch
    g, mask = _problem(afc, elem, n)
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    rhs = np.random.default_rng(n[0] + 7 * n[2]).uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    want, its_want = Gmres(g, afc, mask, nsm).solve(rhs, m, 1e-5, maxit)
    x, its, _ = g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-5, ksp_maxit=maxit,
                                                        gmres_restart=m, precision=afc.AFC_MIXED))
    assert its == its_want
    assert np.array_equal(x, want.astype(np.float64))


@pytest.mark.parametrize("n", [(33, 33, 33), (65, 65, 66)])
def test_stationary_solve_repeats_its_bits(afc, n):
    xyz = W.grid_coords(n)
    g, mask = _problem(afc, "p1", n)
    o = afc.default_opts(limiter=afc.AFC_LIM_MC, omega=0.5, ksp=afc.AFC_KSP_GMRES, ksp_atol=0.0, ksp_rtol=1e-2, fp_tol=1e-12,
                         fp_maxit=60, precision=afc.AFC_MIXED)
    res = []
    for _ in range(2):
        g.set_solution(np.where(mask, xyz[:, 1], 0.0))
        st = g.solve_stationary(o)
        res.append((st["outer_its"], st["inner_its"], g.get_solution().tobytes()))
    assert res[0] == res[1]
