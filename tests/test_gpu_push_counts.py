"""pic_push_counts: the particle slots of pushed chunks and of chunks at rest. Without a field, chunks with power-of-two
particles per cell (whose electrons carry their ions) are at rest; with one on every node, with other particles per cell and
in double precision none is; 1D and 3D contexts have no such counts."""
import ctypes

import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W
from paper_1009_2727_gb300 import capi

pytestmark = pytest.mark.gpu


def dark(ppc, precision="mixed"):
    w = W.shrink(W.stage_2d(5.0), 96, 256, precision=precision)
    w["pml_cells"] = 6
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    w["plasma"].update(ppc_x=ppc, ppc_z=ppc, z_start_lab=5.0 * 120 * dz, ramp_lab=2e-6)
    del w["laser"]
    return w


def counts(w, steps, field=0.0):
    from paper_1009_2727_gb300.pic import Simulation
    sim = Simulation(w, tile=(8, 16), sort_every=16)
    if field:
        for c in range(6):
            sim.set_field(c, np.full(sim.shape, field))
    sim.step(steps)
    sim.sync()
    n = sim.push_counts()
    sim.close()
    return n


def test_chunks_at_rest_are_counted():
    pushed, rest = counts(dark(4), 60)
    assert rest > 10 * pushed
    all_pushed, none = counts(dark(4), 60, field=1e-25)
    assert none == 0 and all_pushed == pushed + rest


@pytest.mark.parametrize("w", [dark(3), dark(2, "fp64")], ids=["ppc3", "fp64"])
def test_always_pushed(w):
    pushed, rest = counts(w, 40)
    assert pushed > 0 and rest == 0


def test_other_dimensions():
    from paper_1009_2727_gb300.pic import Simulation
    sim = Simulation(W.parity_1d())
    a, b = ctypes.c_int64(), ctypes.c_int64()
    assert sim.L.pic_push_counts(sim.h, ctypes.byref(a), ctypes.byref(b)) == capi.PIC_EINVAL
    sim.close()
