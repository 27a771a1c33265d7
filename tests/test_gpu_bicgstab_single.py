"""BiCGStab on single-precision vectors, bit for bit: the solution of a mixed-precision linear solve
equals that of the same iteration in numpy, with the sums a thread forms over its rows (every 512th of
a block's contiguous rows) in single precision and everything beyond in double, whose rounding shows
only where a scalar lies within 1e-16 of a rounding boundary of single precision."""
import math

import numpy as np
import pytest

from test_gpu_gmres_single import F, Gmres, _fma, _problem, afc  # noqa: F401

pytestmark = pytest.mark.gpu


class Bicgstab(Gmres):
    def threads(self, *pairs):
        """Double sums of single-precision thread sums of a * b."""
        N = self.N
        G = max(1, min(-(-N // 64), self.nsm))
        start = np.arange(G + 1) * N // G
        most = int(np.diff(start).max())
        J = -(-most // 512)
        at = start[:-1, None] + np.arange(J * 512)
        use = at < start[1:, None]
        at = np.where(use, at, 0)
        out = []
        for a, b in pairs:
            acc = np.zeros((G, 512), F)
            for j in range(J):
                sl = slice(512 * j, 512 * j + 512)
                acc = np.where(use[:, sl], _fma(a[at[:, sl]], b[at[:, sl]], acc), acc)
            out.append(math.fsum(acc.astype(np.float64).ravel()))
        return out

    def solve(self, rhs, rtol, maxit):
        r = rhs.astype(F)
        rh, p, x, v = r.copy(), r.copy(), np.zeros(self.N, F), np.zeros(self.N, F)
        ph = self.dinv * p
        rho = self.threads((r, r))[0]
        tol, its, tb, to = rtol * math.sqrt(rho), 0, F(0), F(0)
        while True:
            if its:
                p = _fma(tb, _fma(-to, v, p), r)
                ph = self.dinv * p
            v = self.product(ph)
            alpha = rho / self.threads((rh, v))[0]
            ta = F(alpha)
            r = _fma(-ta, v, r)
            sg = self.dinv * r
            its += 1
            if math.sqrt(self.threads((r, r))[0]) < tol:
                return _fma(ta, ph, x), its
            t = self.product(sg)
            ts, tt = self.threads((t, r), (t, t))
            omega = ts / tt
            to = F(omega)
            r = _fma(-to, t, r)
            rr, rhr = self.threads((r, r), (rh, r))
            x = _fma(to, sg, _fma(ta, ph, x))
            tb = F((rhr / rho) * (alpha / omega))
            rho = rhr
            if math.sqrt(rr) < tol or its >= maxit:
                return x, its


# one row a thread (77,121 rows are the last size but a few of that), two to four
@pytest.mark.parametrize("elem,n", [("p1", (9, 8, 7)), ("q1", (41, 33, 57)), ("p1", (57, 57, 57)), ("q1", (65, 65, 65))])
def test_solution_bits(afc, elem, n):  # noqa: F811
    import torch
    g, mask = _problem(afc, elem, n)
    nsm = torch.cuda.get_device_properties(0).multi_processor_count
    rhs = np.random.default_rng(n[0] + 7 * n[2]).uniform(-1.0, 1.0, g.N) * g.lumped_mass()
    want, its_want = Bicgstab(g, afc, mask, nsm).solve(rhs, 1e-5, 8)
    x, its, _ = g.linear_solve(0, rhs, afc.default_opts(ksp=afc.AFC_KSP_BICGSTAB, ksp_atol=0.0, ksp_rtol=1e-5, ksp_maxit=8,
                                                        precision=afc.AFC_MIXED))
    assert its == its_want
    assert np.array_equal(x, want.astype(np.float64))
