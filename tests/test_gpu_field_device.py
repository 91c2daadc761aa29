"""pic_get_field to device memory: the fields are those of the host copy, and memory that the caller's stream still uses
when the allocator hands it out again is not written before that use ends (1D, 2D, 3D; a run on its own stream and on the
caller's, the caller on the default stream and on another one)."""
import numpy as np
import pytest

from paper_1009_2727_gb300 import capi
from paper_1009_2727_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def workload(dim):
    if dim == 1:
        return W.parity_1d()
    return W.shrink(W.parity_2d(), 48, 160) if dim == 2 else W.shrink3(W.parity_3d(), 24, 24, 64)


@pytest.mark.parametrize("own", [False, True], ids=["callers-stream", "own-stream"])
@pytest.mark.parametrize("side", [False, True], ids=["default", "side"])
@pytest.mark.parametrize("dim", [1, 2, 3])
def test_destination_in_use(dim, side, own):
    import torch
    from paper_1009_2727_gb300.pic import Simulation
    cur = torch.cuda.Stream() if side else torch.cuda.default_stream()
    with torch.cuda.stream(cur):
        sim = Simulation(workload(dim), stream=torch.cuda.Stream() if own else cur)
        sim.step(40)
        sim.sync()
        reused = 0
        for comp in (capi.EY, capi.BX, capi.RHO):
            want = sim.field(comp)
            assert np.abs(want).max() > 0
            x = torch.full(sim.shape, 7.0, dtype=torch.float64, device="cuda")
            addr = x.data_ptr()
            torch.cuda.synchronize()
            torch.cuda._sleep(400_000_000)   # about 0.2 s
            y = x + 0.0                      # reads x after the wait
            del x
            t = sim.field_device(comp)
            reused += t.data_ptr() == addr
            torch.cuda.synchronize()
            assert (y == 7.0).all()
            got = t.cpu().numpy()
            if comp == capi.RHO:             # atomic sums in another order
                assert np.abs(got - want).max() <= 1e-10 * 1.6e-19 * sim.w["gamma_boost"] * sim.w["plasma"]["n0"]
            else:
                assert np.array_equal(got, want)
        assert reused
        sim.close()
