"""The work a user of this framework has it do, as cases that can be timed and compared.

Four kinds, each through the public binding (paper_2110_15676_gb300.afc):

* "step": time steps of one transient problem (explicit SSP with Zalesak's limiter, or the
  nonlinear Crank-Nicolson scheme with its fixed point and inner solves), from a state the
  caller holds on the device to a state the caller receives on the device;
* "stationary": one stationary solve with the monolithic limiter (damped fixed point, inner
  Krylov solves), from the initial guess to the converged solution;
* "batch": steps of many independent explicit problems together;
* "serve": a burst of requests (transient and stationary) through the request server, each
  built, solved and returned to host memory.

Grids, coefficients and tolerances are those of the repository's tests and benchmark: box
grids of 9 to 129 nodes per side, P1 (Kuhn) and Q1, eps from 0 to 1e-4, a rotating or a
constant velocity, double precision and the mixed mode.  `exact` computes the same results
in 64 bits with plain torch, from the equations of the method.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2110_15676_gb300 import afc

# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------


def _step(name, elem, n, scheme, precision, steps, field="hump", eps=1e-6):
    c = {"kind": "step", "elem": elem, "nx": n[0], "ny": n[1], "nz": n[2], "scheme": scheme,
         "precision": precision, "steps": steps, "field": field, "eps": eps}
    return {"name": name, **c} if name else c


def _stationary(name, elem, n, precision, ksp, eps=1e-8, tol=1e-12):
    c = {"kind": "stationary", "elem": elem, "nx": n[0], "ny": n[1], "nz": n[2], "precision": precision,
         "ksp": ksp, "eps": eps, "tol": tol}
    return {"name": name, **c} if name else c


def _batch(name, count, lo, hi, elems, precision, steps, mix):
    c = {"kind": "batch", "count": count, "lo": lo, "hi": hi, "elems": elems, "precision": precision,
         "steps": steps, "mix": mix}
    return {"name": name, **c} if name else c


def _serve(name, count, lo, hi, mix):
    c = {"kind": "serve", "count": count, "lo": lo, "hi": hi, "mix": mix}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest problem of the repository's configurations, 20 steps as configured: a
        # step is a dozen launches of a few microseconds
        _step("ssp3_p1_9", "p1", (9, 9, 9), "ssp3", "fp64", 20),
        # an ordinary explicit run on a ragged box, raw fluxes in single precision
        _step("ssp3_q1_41x33x57_mixed", "q1", (41, 33, 57), "ssp3", "mixed", 10),
        # rotating shapes (eps = 0, discontinuous data) on two million nodes, Heun's scheme
        _step("ssp2_q1_129", "q1", (129, 129, 129), "ssp2", "fp64", 2, "shapes", 0.0),
        # Crank-Nicolson with Zalesak's limiter on a small P1 grid (the paper's level 5)
        _step("cn_p1_33", "p1", (33, 33, 33), "cn", "fp64", 3),
        # the benchmark's Crank-Nicolson step (level 6), in double precision and mixed
        _step("cn_q1_65", "q1", (65, 65, 65), "cn", "fp64", 2),
        _step("cn_q1_65_mixed", "q1", (65, 65, 65), "cn", "mixed", 2),
        # stationary monolithic limiting: a small double-precision solve on a ragged box,
        # an ordinary mixed one, and the large grid of the configurations
        _stationary("stationary_q1_27x21x33", "q1", (27, 21, 33), "fp64", "gmres"),
        _stationary("stationary_p1_49", "p1", (49, 49, 49), "mixed", "gmres"),
        _stationary("stationary_p1_129", "p1", (129, 129, 129), "mixed", "gmres", tol=1e-11),
        # batches of independent explicit problems: the configured size range in the mixed
        # mode, and a small double-precision batch of both elements
        _batch("batch_q1_48_mixed", 48, 17, 49, "q1", "mixed", 5, 1),
        _batch("batch_p1q1_12", 12, 9, 33, "p1q1", "fp64", 5, 2),
        # a burst of requests to the server
        _serve("serve_8", 8, 17, 33, 3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("step", "step", "step", "stationary", "stationary", "batch", "serve"))
    elem = rng.choice(("p1", "q1"))
    mix = rng.randrange(1, 1 << 20)
    if kind == "step":
        scheme = rng.choice(("ssp2", "ssp3", "cn"))
        top = 65 if scheme == "cn" else 113
        n = tuple(_log_int(rng, 9, top) for _ in range(3))
        precision = rng.choice(("fp64", "mixed"))
        steps = rng.randint(1, 3) if scheme == "cn" else rng.randint(2, 12)
        return _step(None, elem, n, scheme, precision, steps, rng.choice(("hump", "shapes")),
                     round(10.0 ** rng.uniform(-8.0, -4.0), 12))
    if kind == "stationary":
        n = tuple(_log_int(rng, 13, 57) for _ in range(3))
        return _stationary(None, elem, n, rng.choice(("fp64", "mixed")), rng.choice(("gmres", "gmres", "bicgstab")),
                           round(10.0 ** rng.uniform(-8.0, -4.0), 12))
    if kind == "batch":
        hi = rng.randint(20, 49)
        return _batch(None, rng.randint(3, 48), rng.randint(9, 17), hi, rng.choice(("p1", "q1", "p1q1")),
                      rng.choice(("fp64", "mixed")), rng.randint(2, 6), mix)
    return _serve(None, rng.randint(3, 8), 17, rng.randint(20, 33), mix)


# ---------------------------------------------------------------------------
# inputs (host arrays, as a user's program builds them)
# ---------------------------------------------------------------------------

CFL_SSP, CFL_CN = 0.5, 1.0
FP_TOL_CN, KSP_ATOL = 1e-10, 1e-12
FP_TOL_SERVE, FP_MAXIT_ST, OMEGA_ST, RTOL_ST = 1e-12, 1500, 0.5, 1e-2


def _coords(n):
    xs = [np.linspace(0.0, 1.0, k) for k in n]
    z, y, x = np.meshgrid(xs[2], xs[1], xs[0], indexing="ij")
    return np.stack([x.ravel(), y.ravel(), z.ravel()], axis=1)


def _faces(n):
    iz, iy, ix = np.meshgrid(np.arange(n[2]), np.arange(n[1]), np.arange(n[0]), indexing="ij")
    return ix.ravel(), iy.ravel(), iz.ravel()


def _boundary(n):
    ix, iy, iz = _faces(n)
    return ((ix == 0) | (ix == n[0] - 1) | (iy == 0) | (iy == n[1] - 1) | (iz == 0) | (iz == n[2] - 1)).astype(np.uint8)


def _hump(xyz, center, radius=0.15):
    r = np.sqrt(((xyz - center) ** 2).sum(axis=1))
    return np.where(r <= radius, 0.5 * (1.0 + np.cos(np.pi * np.minimum(r, radius) / radius)), 0.0)


def _transient_data(elem, n, eps, field, rng):
    """A transient problem: rotating velocity, a hump or the three bodies, zero Dirichlet data."""
    xyz = _coords(n)
    turn = rng.uniform(0.8, 1.25)
    b = turn * np.stack([0.5 - xyz[:, 1], xyz[:, 0] - 0.5, np.zeros(len(xyz))], axis=1)
    phi = rng.uniform(0.0, 2.0 * np.pi)
    at = np.array([0.5 + 0.25 * math.cos(phi), 0.5 + 0.25 * math.sin(phi), 0.5])
    if field == "hump":
        u0 = _hump(xyz, at)
    else:   # a cube, a cone and a hollow cylinder, turned by phi about the axis
        c, s = math.cos(phi), math.sin(phi)
        x = 0.5 + c * (xyz[:, 0] - 0.5) + s * (xyz[:, 1] - 0.5)
        y = 0.5 - s * (xyz[:, 0] - 0.5) + c * (xyz[:, 1] - 0.5)
        z = xyz[:, 2]
        tall = (z >= 0.25) & (z <= 0.75)
        cube = (np.abs(x - 0.5) <= 0.125) & (np.abs(y - 0.25) <= 0.125) & (np.abs(z - 0.5) <= 0.125)
        cone = tall & (np.hypot(x - 0.75, y - 0.5) <= 0.125 * (1.0 - (z - 0.25) / 0.5))
        rh = np.hypot(x - 0.5, y - 0.75)
        u0 = (cube | cone | (tall & (rh >= 0.0625) & (rh <= 0.125))).astype(np.float64)
    mask = _boundary(n)
    return {"elem": elem, "n": n, "eps": eps, "c": 0.0, "b": b, "f": np.zeros(len(xyz)),
            "u0": np.where(mask != 0, 0.0, u0), "mask": mask, "ud": np.zeros(len(xyz))}


def _random_transient(elem, n, rng, c=0.0):
    """A batched or served instance: unit constant velocity, eps log-uniform, a hump somewhere."""
    xyz = _coords(n)
    v = rng.normal(size=3)
    v /= np.linalg.norm(v)
    mask = _boundary(n)
    u0 = _hump(xyz, rng.uniform(0.3, 0.7, size=3))
    return {"elem": elem, "n": n, "eps": float(10.0 ** rng.uniform(-8.0, -4.0)), "c": c,
            "b": np.tile(v, (len(xyz), 1)), "f": np.zeros(len(xyz)), "u0": np.where(mask != 0, 0.0, u0),
            "mask": mask, "ud": np.zeros(len(xyz))}


def _stationary_data(elem, n, eps, rng):
    """The inflow problem: b near (1, -0.5, 0.25), a source block, discontinuous inflow data."""
    xyz = _coords(n)
    ix, iy, iz = _faces(n)
    x, y, z = xyz.T
    inflow = (ix == 0) | (iy == n[1] - 1) | (iz == 0)
    ud = np.where((ix == 0) & (y < rng.uniform(0.4, 0.6)), 1.0, 0.0)
    lo = rng.uniform(0.2, 0.3)
    f = np.where((x >= lo) & (x <= lo + 0.25) & (y >= lo) & (y <= lo + 0.25) & (z >= lo) & (z <= lo + 0.25), 1.0, 0.0)
    b = np.array([1.0, -0.5, 0.25]) * rng.uniform(0.9, 1.1, size=3)
    return {"elem": elem, "n": n, "eps": eps, "c": float(rng.uniform(0.8, 1.0)), "b": np.tile(b, (len(xyz), 1)),
            "f": f, "u0": np.where(inflow, ud, 0.0), "mask": inflow.astype(np.uint8), "ud": ud}


def _data(case, seed):
    """The host data of every problem of a case, in order, with what each is ("transient" or "stationary")."""
    rng = np.random.default_rng([int(seed), 2110])
    kind = case["kind"]
    if kind in ("step", "stationary"):
        n = (case["nx"], case["ny"], case["nz"])
        if kind == "step":
            return [("transient", _transient_data(case["elem"], n, case["eps"], case["field"], rng))]
        return [("stationary", _stationary_data(case["elem"], n, case["eps"], rng))]
    sizes = np.random.default_rng([int(case["mix"]), 15676])
    out = []
    for q in range(case["count"]):
        n = (int(sizes.integers(case["lo"], case["hi"] + 1)),) * 3
        if kind == "batch":
            elem = case["elems"] if case["elems"] != "p1q1" else ("p1", "q1")[q % 2]
            out.append(("transient", _random_transient(elem, n, rng)))
        else:   # transient and stationary, P1 and Q1 in turn
            elem = ("p1", "q1")[(q // 2) % 2]
            if q % 2 == 0:
                out.append(("transient", _random_transient(elem, n, rng, c=float(rng.uniform(0.0, 1.0)))))
            else:
                out.append(("stationary", _stationary_data(elem, n, float(10.0 ** rng.uniform(-8.0, -4.0)), rng)))
    return out


SERVE_STEPS = 20


# ---------------------------------------------------------------------------
# the framework's side
# ---------------------------------------------------------------------------


def _problem(d, family, precision):
    p = afc.Problem.structured(d["elem"], d["n"])
    p.set_coefficients(d["eps"], d["b"], d["c"], d["f"])
    p.set_dirichlet(d["mask"], d["ud"])
    p.assemble(family, precision)
    return p


def _precision(case):
    return afc.AFC_MIXED if case.get("precision") == "mixed" else afc.AFC_FP64


def _stationary_opts(precision, ksp, tol):
    gm = ksp == "gmres"
    return afc.default_opts(limiter=afc.AFC_LIM_MC, omega=OMEGA_ST, ksp=afc.AFC_KSP_GMRES if gm else afc.AFC_KSP_BICGSTAB,
                            gmres_restart=20, ksp_atol=0.0, ksp_rtol=RTOL_ST, fp_tol=tol, fp_maxit=FP_MAXIT_ST,
                            precision=precision)


def prepare(case, seed):
    data = _data(case, seed)
    kind, prec = case["kind"], _precision(case)
    if kind == "step":
        d = data[0][1]
        cn = case["scheme"] == "cn"
        p = _problem(d, afc.AFC_FAMILY_FCT, prec)
        dt = p.cfl_timestep(CFL_CN if cn else CFL_SSP)
        scheme = {"ssp2": afc.AFC_SSP2, "ssp3": afc.AFC_SSP3, "cn": afc.AFC_CN_NONLINEAR}[case["scheme"]]
        inner = {"ksp_atol": 0.0, "ksp_rtol": 1e-6} if prec == afc.AFC_MIXED else {"ksp_atol": KSP_ATOL}
        opts = afc.default_opts(scheme=scheme, dt=dt, fp_tol=FP_TOL_CN, precision=prec, **(inner if cn else {}))
        u0 = torch.tensor(d["u0"], device="cuda")
        return {"kind": kind, "p": p, "opts": opts, "steps": case["steps"], "u0": u0, "u": torch.empty_like(u0)}
    if kind == "stationary":
        d = data[0][1]
        p = _problem(d, afc.AFC_FAMILY_MC, prec)
        u0 = torch.tensor(d["u0"], device="cuda")
        return {"kind": kind, "p": p, "opts": _stationary_opts(prec, case["ksp"], case["tol"]), "u0": u0, "u": torch.empty_like(u0)}
    if kind == "batch":
        ps = [_problem(d, afc.AFC_FAMILY_FCT, prec) for _, d in data]
        u0 = [torch.tensor(d["u0"], device="cuda") for _, d in data]
        return {"kind": kind, "ps": ps, "batch": afc.Batch(ps), "dt": [p.cfl_timestep(CFL_SSP) for p in ps],
                "opts": afc.default_opts(scheme=afc.AFC_SSP3, precision=prec), "steps": case["steps"], "u0": u0,
                "u": [torch.empty_like(u) for u in u0]}
    reqs = []
    for what, d in data:
        if what == "transient":
            reqs.append(afc.Request(afc.AFC_REQ_TRANSIENT, d["elem"], d["n"], d["eps"], d["c"], d["b"], d["u0"], d["mask"],
                                    d["ud"], f=d["f"], steps=SERVE_STEPS, cfl=CFL_SSP,
                                    opts=afc.default_opts(scheme=afc.AFC_SSP3, precision=afc.AFC_MIXED)))
        else:
            reqs.append(afc.Request(afc.AFC_REQ_STATIONARY, d["elem"], d["n"], d["eps"], d["c"], d["b"], d["u0"], d["mask"],
                                    d["ud"], f=d["f"], opts=_stationary_opts(afc.AFC_MIXED, "gmres", FP_TOL_SERVE)))
    return {"kind": kind, "server": afc.Server(), "reqs": reqs}


def run(state):
    kind = state["kind"]
    if kind == "step":
        p, opts = state["p"], state["opts"]
        p.set_solution(state["u0"])
        for _ in range(state["steps"]):
            p.step(opts)
        return p.get_solution(state["u"])
    if kind == "stationary":
        p = state["p"]
        p.set_solution(state["u0"])
        p.solve_stationary(state["opts"])
        return p.get_solution(state["u"])
    if kind == "batch":
        for p, u in zip(state["ps"], state["u0"]):
            p.set_solution(u)
        state["batch"].step(state["opts"], dt=state["dt"], nsteps=state["steps"])
        return [p.get_solution(u) for p, u in zip(state["ps"], state["u"])]
    server = state["server"]
    ids = [server.submit(r) for r in state["reqs"]]
    out = []
    for i in ids:
        out.append(server.wait(i)[1])
        server.release(i)
    return out


# ---------------------------------------------------------------------------
# the work of a pass
# ---------------------------------------------------------------------------

# Nominal counts per case kind, at the tolerances above: fixed-point corrections and Krylov
# iterations of a Crank-Nicolson step and of a stationary solve.
CN_CORRECTIONS, CN_KRYLOV = 13, 48
ST_CORRECTIONS, ST_KRYLOV = 600, 5000


def _stage_work(elem, N, mixed):
    """One explicit stage: the low-order operator, the pair data and about ten node vectors once."""
    K, E = (15, 7) if elem == "p1" else (27, 13)
    pair = 8 if mixed else 16
    return N * (8.0 * K + pair * E + 80.0), N * (2.0 * K + 2.0 * 10.0 * E + 30.0)


def work(case):
    kind = case["kind"]
    b = f = 0.0
    mixed = case.get("precision") == "mixed"
    if kind == "step":
        N = case["nx"] * case["ny"] * case["nz"]
        K, E = (15, 7) if case["elem"] == "p1" else (27, 13)
        if case["scheme"] == "cn":
            it = N * ((4.0 if mixed else 8.0) * 2 * K + (4.0 if mixed else 8.0) * 14)
            cor = N * (8.0 * K + 16.0 * E + 80.0)
            b = CN_KRYLOV * it + CN_CORRECTIONS * cor
            f = CN_KRYLOV * N * (4.0 * K + 26.0) + CN_CORRECTIONS * N * (2.0 * K + 10.0 * E)
        else:
            sb, sf = _stage_work(case["elem"], N, mixed)
            ns = 2 if case["scheme"] == "ssp2" else 3
            b, f = ns * sb, ns * sf
        return {"bytes": case["steps"] * b + 16.0 * N, "flops": case["steps"] * f}
    if kind == "stationary":
        N = case["nx"] * case["ny"] * case["nz"]
        return dict(zip(("bytes", "flops"), _stationary_work(case["elem"], N, mixed)))
    for what, d in _shapes(case):
        N = d[1] ** 3
        if what == "transient":
            sb, sf = _stage_work(d[0], N, mixed or kind == "serve")
            steps = SERVE_STEPS if kind == "serve" else case["steps"]
            b += 3 * steps * sb
            f += 3 * steps * sf
        else:
            sb, sf = _stationary_work(d[0], N, True)
            b += sb
            f += sf
    return {"bytes": b, "flops": f}


def _stationary_work(elem, N, mixed):
    K, E = (15, 7) if elem == "p1" else (27, 13)
    w = 4.0 if mixed else 8.0
    it = N * (w * K + w * 25.0)
    cor = N * (8.0 * K + 16.0 * E + 60.0)
    return (ST_KRYLOV * it + ST_CORRECTIONS * cor,
            ST_KRYLOV * N * (2.0 * K + 42.0) + ST_CORRECTIONS * N * (2.0 * K + 14.0 * E))


def _shapes(case):
    sizes = np.random.default_rng([int(case["mix"]), 15676])
    out = []
    for q in range(case["count"]):
        n = int(sizes.integers(case["lo"], case["hi"] + 1))
        if case["kind"] == "batch":
            out.append(("transient", (case["elems"] if case["elems"] != "p1q1" else ("p1", "q1")[q % 2], n)))
        else:
            out.append((("transient", "stationary")[q % 2], (("p1", "q1")[(q // 2) % 2], n)))
    return out


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------


class _Exact:
    """Matrices of one problem by diagonals (one row of `K` values per node) and the method on them."""

    def __init__(self, d, family):
        dev = "cuda" if torch.cuda.is_available() else "cpu"
        nx, ny, nz = d["n"]
        self.n, self.N = d["n"], nx * ny * nz
        h = [1.0 / (k - 1) for k in d["n"]]
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        corners = [(k & 1, (k >> 1) & 1, k >> 2) for k in range(8)]
        if d["elem"] == "q1":
            cells = [corners]
        else:   # Kuhn: one path from corner (0,0,0) to (1,1,1) per order of the axes
            cells = []
            for a, c, e in ((0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)):
                path = [[0, 0, 0]]
                for ax in (a, c, e):
                    path.append(list(path[-1]))
                    path[-1][ax] = 1
                cells.append([tuple(v) for v in path])
        offs = sorted({tuple(b[x] - a[x] for x in range(3)) for ty in cells for a in ty for b in ty},
                      key=lambda o: o[0] + nx * (o[1] + ny * o[2]))
        self.o = [o[0] + nx * (o[1] + ny * o[2]) for o in offs]
        self.K, self.pad = len(offs), max(self.o)
        at = {o: k for k, o in enumerate(offs)}
        shape = (self.K, nz, ny, nx)
        M, S, C = (torch.zeros(shape, dtype=torch.float64, device=dev) for _ in range(3))
        mask = torch.zeros(shape, dtype=torch.bool, device=dev)
        B = t(d["b"]).T.reshape(3, nz, ny, nx)
        cut = lambda v: (slice(v[2], nz - 1 + v[2]), slice(v[1], ny - 1 + v[1]), slice(v[0], nx - 1 + v[0]))  # noqa: E731
        for ty in cells:
            for a, va in enumerate(ty):
                for b, vb in enumerate(ty):
                    k = at[tuple(vb[x] - va[x] for x in range(3))]
                    rows = (k, *cut(va))
                    m, s, conv = _q1_entry(va, vb, ty, h) if d["elem"] == "q1" else _p1_entry(ty, a, b, h)
                    M[rows] += m
                    S[rows] += s
                    mask[rows] = True
                    for j, w in enumerate(conv):
                        for x in range(3):
                            if w[x]:
                                C[rows] += w[x] * B[(x, *cut(ty[j]))]
        M, S, C, mask = (v.reshape(self.K, self.N) for v in (M, S, C, mask))
        self.M, self.mask, mid = M, mask, self.K // 2
        self.mL = M.sum(0)
        self.f = self.mL * t(d["f"])
        self.dir, self.ud, self.u0 = t(d["mask"]) != 0, t(d["ud"]), t(d["u0"])
        A = d["eps"] * S + C + d["c"] * M if family == "fct" else C
        D = -torch.clamp(torch.maximum(A, self.mirror(A)), min=0.0) * mask
        D[mid] = 0.0
        D[mid] = -D.sum(0)
        self.D = D
        self.AA = A + D
        if family == "mc":
            self.AA = self.AA + d["eps"] * S
            self.AA[mid] += d["c"] * self.mL
            self.C, self.CT = C, self.mirror(C)
        self.mid = mid
        self.free = ~self.dir
        self.off = mask.clone()
        self.off[mid] = False
        del S

    def around(self, v):
        """Row k: the values of v at the neighbours i + o_k (0 outside)."""
        p = torch.nn.functional.pad(v, (self.pad, self.pad))
        return torch.stack([p[self.pad + o: self.pad + o + self.N] for o in self.o])

    def mirror(self, A):
        """Row k: a_ji of the pair (i, j = i + o_k)."""
        rows = []
        for k, o in enumerate(self.o):
            p = torch.nn.functional.pad(A[self.K - 1 - k], (self.pad, self.pad))
            rows.append(p[self.pad + o: self.pad + o + self.N])
        return torch.stack(rows)

    def mul(self, A, v):
        p = torch.nn.functional.pad(v, (self.pad, self.pad))
        y = A[0] * p[self.pad + self.o[0]: self.pad + self.o[0] + self.N]
        for k in range(1, self.K):
            y.addcmul_(A[k], p[self.pad + self.o[k]: self.pad + self.o[k] + self.N])
        return y

    def dt(self, cfl):
        return cfl * float((self.mL / self.AA[self.mid])[self.free].min())

    def bounds(self, v):
        V = self.around(v)
        big = torch.where(self.mask, V, torch.full_like(V, -math.inf)).amax(0)
        small = torch.where(self.mask, V, torch.full_like(V, math.inf)).amin(0)
        return big, small

    def zalesak(self, r, ut, dt):
        """F* = sum_j alpha_ij r_ij with the bounds of the predictor ut."""
        Pp, Pm = r.clamp(min=0.0).sum(0), r.clamp(max=0.0).sum(0)
        big, small = self.bounds(ut)
        one = torch.ones_like(ut)
        Rp = torch.where((Pp == 0) | self.dir, one, torch.minimum(one, self.mL * (big - ut) / dt / torch.where(Pp == 0, one, Pp)))
        Rm = torch.where((Pm == 0) | self.dir, one, torch.minimum(one, self.mL * (small - ut) / dt / torch.where(Pm == 0, one, Pm)))
        alpha = torch.where(r > 0, torch.minimum(Rp, self.around(Rm)), torch.minimum(Rm, self.around(Rp)))
        return torch.where(self.dir, torch.zeros_like(ut), (alpha * r).sum(0))

    def stage(self, u, dt):
        zero = torch.zeros_like(u)
        rate = torch.where(self.dir, zero, (self.f - self.mul(self.AA, u)) / self.mL)
        ut = torch.where(self.dir, self.ud, u + dt * rate)
        r = torch.where(self.off, self.M * (rate - self.around(rate)) + self.D * (self.around(u) - u), 0.0)
        return torch.where(self.dir, self.ud, ut + dt * self.zalesak(r, ut, dt) / self.mL)

    def ssp(self, u, dt, stages):
        if stages == 2:
            return 0.5 * (u + self.stage(self.stage(u, dt), dt))
        a = 0.75 * u + 0.25 * self.stage(self.stage(u, dt), dt)
        return u / 3.0 + 2.0 / 3.0 * self.stage(a, dt)

    def system(self, scale, dt):
        B = scale * self.AA
        if dt:
            B[self.mid] += self.mL / dt
        B[:, self.dir] = 0.0
        B[self.mid, self.dir] = 1.0
        return B

    def solve(self, B, rhs, atol, rtol):
        """Jacobi-preconditioned BiCGStab."""
        di, x, r = 1.0 / B[self.mid], torch.zeros_like(rhs), rhs.clone()
        rh, p, v = r.clone(), torch.zeros_like(r), torch.zeros_like(r)
        rho = alpha = om = torch.ones((), dtype=torch.float64, device=r.device)
        tol = max(atol, rtol * float(r.norm()))
        for _ in range(2000):
            if float(r.norm()) < tol:
                break
            new = rh.dot(r)
            p = r + (new / rho) * (alpha / om) * (p - om * v)
            v = self.mul(B, di * p)
            alpha = new / rh.dot(v)
            s = r - alpha * v
            x = x + alpha * di * p
            if float(s.norm()) < tol:
                break
            t = self.mul(B, di * s)
            om = t.dot(s) / t.dot(t)
            x = x + om * di * s
            r = s - om * t
            rho = new
        return x

    def cn(self, u_old, dt):
        y = self.mul(self.AA, u_old)
        ut = torch.where(self.dir, self.ud, u_old - 0.5 * dt * (y - self.f) / self.mL)
        b0 = self.mL / dt * u_old - 0.5 * y + self.f
        B = self.system(0.5, dt)
        u = torch.where(self.dir, self.ud, u_old)
        for _ in range(100):
            a, s = u - u_old, u + u_old
            q = torch.where(self.off, self.D * (self.around(s) - s), 0.0)
            r = torch.where(self.off, self.M / dt * (a - self.around(a)) + 0.5 * q, 0.0)
            same = (r > 0) & (q > 0) | (r < 0) & (q < 0)
            r = torch.where(same, torch.where(r.abs() < q.abs(), r, q), torch.zeros_like(r))
            res = b0 + self.zalesak(r, ut, dt) - (self.mL / dt * u + 0.5 * self.mul(self.AA, u))
            res = torch.where(self.dir, torch.zeros_like(res), res)
            if float(res.norm()) < math.sqrt(self.N) * FP_TOL_CN:
                break
            u = u + self.solve(B, res, KSP_ATOL, 0.0)
        return u

    def mc_flux(self, u):
        """F* of the monolithic convex limiter."""
        U, d = self.around(u), self.D
        big, small = self.bounds(u)
        live = self.off & (d != 0)
        two = torch.where(live, 2.0 * d, torch.ones_like(d))
        r = torch.where(live, d * (U - u), 0.0)
        bar = torch.where(live, (d * (U + u) + self.C * (U - u)) / two, 0.0)
        rab = torch.where(live, (d * (U + u) - self.CT * (U - u)) / two, 0.0)
        up = torch.minimum(r, torch.minimum(two * (bar - big), two * (self.around(small) - rab)))
        dn = torch.maximum(r, torch.maximum(two * (bar - small), two * (self.around(big) - rab)))
        return torch.where(live, torch.where(r > 0, up, dn), 0.0).sum(0)

    def stationary(self, u0, tol):
        B = self.system(1.0, 0.0)
        u = torch.where(self.dir, self.ud, u0)
        for _ in range(FP_MAXIT_ST):
            res = torch.where(self.dir, 0.0, self.f + self.mc_flux(u) - self.mul(self.AA, u))
            if float(res.norm()) < math.sqrt(self.N) * tol:
                break
            u = u + OMEGA_ST * self.solve(B, res, 0.0, RTOL_ST)
        return u


def _line(a, b):
    """Integrals on [0, 1] of l_a l_b and of l_a l_b' for the two linear functions."""
    return (1.0 / 3.0 if a == b else 1.0 / 6.0), (0.5 if b else -0.5)


def _triple(a, j, b):
    return 0.25 if a == j == b else 1.0 / 12.0


def _q1_entry(va, vb, ty, h):
    """(phi_b, phi_a), (grad phi_b, grad phi_a) and, per corner j, the weights of b_j in (b . grad phi_b, phi_a)."""
    m = [_line(va[x], vb[x])[0] * h[x] for x in range(3)]
    g = [(1.0 if va[x] == vb[x] else -1.0) / h[x] for x in range(3)]
    s = g[0] * m[1] * m[2] + m[0] * g[1] * m[2] + m[0] * m[1] * g[2]
    conv = []
    for vj in ty:
        w = []
        for x in range(3):
            p = 1.0
            for y in range(3):
                if y == x:   # l_a l_j l_b', with l_b' = +-1 / h
                    p *= _line(va[y], vj[y])[0] * (1.0 if vb[y] else -1.0)
                else:
                    p *= _triple(va[y], vj[y], vb[y]) * h[y]
            w.append(p)
        conv.append(w)
    return m[0] * m[1] * m[2], s, conv


def _p1_entry(ty, a, b, h):
    """The same for the tetrahedron that walks the axes along the path `ty`."""
    V = h[0] * h[1] * h[2] / 6.0
    axes = [next(x for x in range(3) if ty[q + 1][x] != ty[q][x]) for q in range(3)]
    G = [[0.0] * 3 for _ in range(4)]   # lambda_q = x_{q-1}/h - x_q/h along the path
    for q, ax in enumerate(axes):
        G[q][ax] -= 1.0 / h[ax]
        G[q + 1][ax] += 1.0 / h[ax]
    m = V * (2.0 if a == b else 1.0) / 20.0
    s = V * sum(G[a][x] * G[b][x] for x in range(3))
    conv = [[V * (2.0 if a == j else 1.0) / 20.0 * G[b][x] for x in range(3)] for j in range(4)]
    return m, s, conv


def exact(case, seed):
    if case["kind"] == "stationary" and case["nx"] * case["ny"] * case["nz"] > 400000:
        return None   # hundreds of corrections on two million nodes: too long here
    out = []
    for what, d in _data(case, seed):
        x = _Exact(d, "fct" if what == "transient" else "mc")
        if what == "stationary":
            out.append(x.stationary(x.u0, case.get("tol", FP_TOL_SERVE)))
            continue
        u, cn = x.u0, case.get("scheme") == "cn"
        dt = x.dt(CFL_CN if cn else CFL_SSP)
        for _ in range(SERVE_STEPS if case["kind"] == "serve" else case["steps"]):
            u = x.cn(u, dt) if cn else x.ssp(u, dt, 2 if case.get("scheme") == "ssp2" else 3)
        out.append(u)
        del x
    if case["kind"] == "serve":
        return [u.cpu().numpy() for u in out]
    return out if case["kind"] == "batch" else out[0]
