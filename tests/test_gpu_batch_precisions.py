"""One batch stepped in double, then mixed, then in double again with the same time steps gives the
bits of its instances run alone: its instance table holds the single-precision arrays, which the
first mixed call makes, from then on."""
import numpy as np
import pytest

from paper_2110_15676_gb300 import workloads as W
from pairs import gpu_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", ["per_pass", "per_stage", "per_step"])
def test_batch_changes_its_precision(shape):
    from paper_2110_15676_gb300 import afc
    rng = np.random.default_rng(11)
    wls = [W.random_transient(rng, ("q1", "p1")[q % 2], (6, 12)) for q in range(5)]

    def problems():
        out = []
        for wl in wls:
            g = gpu_problem(wl.elem, wl.n, wl.b, wl.eps, wl.c, wl.f, wl.dir_mask, wl.u_dir)
            g.set_solution(wl.u0)
            out.append(g)
        return out

    gs, solo = problems(), problems()
    dts = [g.cfl_timestep(0.5) for g in gs]
    batch = afc.Batch(gs)
    batch.set_tuning({"per_pass": afc.AFC_BATCH_PER_PASS, "per_stage": afc.AFC_BATCH_PER_STAGE,
                      "per_step": afc.AFC_BATCH_PER_STEP}[shape], 128)
    for prec in (afc.AFC_FP64, afc.AFC_MIXED, afc.AFC_FP64):
        batch.step(afc.default_opts(scheme=afc.AFC_SSP3, precision=prec), dt=dts, nsteps=2)
        for g, s, dt in zip(gs, solo, dts):
            for _ in range(2):
                s.step(afc.default_opts(scheme=afc.AFC_SSP3, dt=dt, precision=prec))
            assert np.array_equal(g.get_solution(), s.get_solution())
