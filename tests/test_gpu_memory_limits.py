"""What a run needs of device memory: scratch that only makes steps faster is not among it. The allocator callback grants
memory up to a limit (or refuses chosen requests); the run must be made, step and agree with one that has all it asks for."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import capi
from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu


class Limited:
    """allocator callbacks on torch's allocator; `refuse(self, n)` decides"""

    def __init__(self, refuse=lambda self, n: False):
        import torch
        self.live, self.asked, self.refuse = {}, [], refuse

        def alloc(n, stream, user):
            self.asked.append(n)
            if self.refuse(self, n):
                return None
            p = torch.cuda.caching_allocator_alloc(int(n), 0, stream)
            self.live[p] = n
            return p

        def free(p, n, stream, user):
            del self.live[p]
            torch.cuda.caching_allocator_delete(p)

        self.cb = capi.ALLOC_FN(alloc), capi.FREE_FN(free)

    def total(self):
        return sum(self.live.values())


def simulation(w, lim, monkeypatch, **kw):
    from paper_1009_2727_gb300 import pic
    monkeypatch.setattr(pic, "torch_allocator", lambda index: lim.cb)
    return pic.Simulation(w, **kw)


def fields(sim):
    return np.stack([sim.field(c) for c in range(6)])


def close(a, b, tol):
    return all(np.linalg.norm(x - y) <= tol * np.linalg.norm(y) for x, y in ((a[:3], b[:3]), (a[3:], b[3:])))


def wide_workload():
    w = W.shrink(W.stage_2d(5.0), 160, 320)
    w.update(precision="fp64", filter_strides=[1, 2], pml_cells=6, particle_guard=24)
    dz = (1.0 + np.sqrt(1 - 1 / 25.0)) * 5.0 * w["dz_lab"]
    w["laser"].update(z_antenna=34 * dz, t_peak=4e-15)
    w["plasma"].update(ppc_x=2, ppc_z=2, z_start_lab=5.0 * 38 * dz)
    return w


def test_wide_filter_with_the_memory_of_a_narrow_one(monkeypatch):
    w = wide_workload()
    lim = Limited()
    sim = simulation(dict(w, filter_strides=[], filter_stride=1), lim, monkeypatch)
    sim.step(1)
    narrow = lim.total()
    sim.close()
    free = Limited()
    a = simulation(w, free, monkeypatch)
    a.step(30)
    # the two-pass kernels' scratch: nine node arrays
    assert free.total() > narrow + 8 * 9 * 161 * 320
    lim = Limited(lambda s, n: s.total() + n > narrow)
    b = simulation(w, lim, monkeypatch)
    b.step(30)
    b.sync()
    fa, fb = fields(a), fields(b)
    assert np.abs(fa).max() > 0 and close(fb, fa, 1e-10)
    a.close()
    b.close()
    assert not free.live and not lim.live


def test_wide_scratch_is_given_back(monkeypatch):
    """an accessor that finds no memory takes the filter's scratch; the run goes on with the tile kernels"""
    w = wide_workload()
    w["plasma"].update(ppc_x=1, ppc_z=1)     # the accessor's scratch is less than the filter's
    lim = Limited()
    sim = simulation(w, lim, monkeypatch)
    ref = simulation(w, Limited(), monkeypatch)
    for s in (sim, ref):
        s.step(15)
    before = lim.total()
    lim.refuse = lambda s, n: s.total() + n > before
    n = len(sim.particles(capi.ELECTRONS)["id"])
    assert n > 0 and lim.total() < before - 8 * 9 * 161 * 320
    for s in (sim, ref):
        s.step(15)
        s.sync()
    assert close(fields(sim), fields(ref), 1e-10)
    sim.close()
    ref.close()
    assert not lim.live


def test_3d_sort_counts_need_no_memory_of_their_own(monkeypatch):
    w = W.shrink3(W.stage_3d(), 128, 128, 255, theta=0.5, precision="mixed")
    lim = Limited()
    sim = simulation({k: v for k, v in w.items() if k not in ("plasma", "laser")}, lim, monkeypatch)
    node_array = 4 * 129 * 129 * 256
    # E, B, J, E^{n-1}, E-bar, two gather copies, the filter's two scratch arrays, twelve split parts; tables
    assert lim.total() <= 35.2 * node_array
    sim.close()


def test_3d_shared_filter_scratch_refused(monkeypatch):
    w = W.shrink3(W.parity_3d(), 24, 24, 64)
    ref = simulation(w, Limited(), monkeypatch)
    array = 8 * 25 * 25 * 80
    # the first request of six node arrays is the filter's
    lim = Limited(lambda s, n: n >= 6 * array and sum(v >= 6 * array for v in s.asked) == 1)
    sim = simulation(w, lim, monkeypatch)
    assert sum(v >= 6 * array for v in lim.asked) == 3
    for s in (sim, ref):
        s.step(20)
        s.sync()
    a, b = fields(sim), fields(ref)
    assert np.abs(b).max() > 0 and close(a, b, 1e-10)
    sim.close()
    ref.close()
