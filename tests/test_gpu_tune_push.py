"""The autotuner's trials push every chunk: on a stage that no pulse has reached yet, where a run's push only moves boxes,
their time per step is that of a push that works (on this box of 3.3 million electrons the push is most of it), while the
tuned run itself still leaves its resting chunks out. On a window that the caller names, the trials are the run's own steps,
and a layout found without a pulse is not handed to a run with one."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def dark(nz):
    w = W.shrink(W.stage_2d(), 256, nz, precision="mixed")
    w["plasma"].update(ppc_x=4, ppc_z=4)
    del w["laser"]
    return w


def ms_per_step(sim, steps=16):
    import torch
    sim.step(4)
    sim.sync()
    a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    a.record()
    sim.step(steps)
    b.record()
    torch.cuda.synchronize()
    return a.elapsed_time(b) / steps


def test_single_run():
    from paper_1009_2727_gb300.pic import Simulation
    sim = Simulation(dark(1024), tune=True)
    own = min(ms_per_step(sim) for _ in range(3))
    pushed, rest = sim.push_counts()
    sim.close()
    assert rest > pushed and sim.tuned["ms_per_step"] > 1.4 * own, (sim.tuned["ms_per_step"], own)


def test_ensemble():
    from paper_1009_2727_gb300.pic import Ensemble
    ens = Ensemble([dark(512), dark(640)], tune="ensemble")
    own = min(ms_per_step(ens) for _ in range(3))
    pushed, rest = np.sum([m.push_counts() for m in ens.members], axis=0)
    tuned = ens.tuned[0]["ms_per_step"]
    ens.close()
    assert rest > pushed and tuned > 1.4 * own, (tuned, own)


def test_window_of_the_run():
    from paper_1009_2727_gb300.pic import Simulation, autotune
    w = dark(1024)
    t = autotune(w, warm=8, steps=16)
    sim = Simulation(w, tile=t["tile"], sort_every=t["sort_every"])
    own = min(ms_per_step(sim) for _ in range(3))
    sim.close()
    assert not t["cached"] and t["ms_per_step"] < 1.4 * own, (t["ms_per_step"], own)
    assert autotune(w, warm=8, steps=16)["cached"]
    lit = dict(w, laser=W.shrink(W.stage_2d(), 256, 1024)["laser"])
    assert not autotune(lit, warm=8, steps=16)["cached"]
