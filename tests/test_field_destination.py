"""Which destinations of pic_get_field(on_device) a kernel writes in place: the context's own GPU's memory, aligned; the rest
goes through a copy, which reaches more (another GPU without a peer mapping) and refuses the rest without a fault. The rule
is compiled for the host and asked for every kind of pointer; on a GPU, pinned host memory and an odd address come out as
the host copy does."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1009_2727_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cstdio>
#include "pic_dst.h"
int main() {
  const cudaMemoryType types[4] = {cudaMemoryTypeUnregistered, cudaMemoryTypeHost, cudaMemoryTypeDevice, cudaMemoryTypeManaged};
  for (int t = 0; t < 4; t++)
    for (int dev = 0; dev < 2; dev++)
      for (int odd = 0; odd < 2; odd++) {
        cudaPointerAttributes a{};
        a.type = types[t];
        a.device = dev;
        printf("%d", (int)picgb::writable_in_place((void*)(size_t)(4096 + 4 * odd), a, 0));
      }
  printf("\n");
}
"""


def test_rule(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src = tmp_path / "dst.cu"
    src.write_text(PROGRAM)
    exe = tmp_path / "dst"
    subprocess.run([nvcc, "-std=c++17", "-I", os.path.join(ROOT, "paper_1009_2727_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.strip()
    # device memory of the context's own GPU, aligned
    assert out == "0000" + "0000" + "1000" + "0000"


@pytest.mark.gpu
@pytest.mark.parametrize("dim", [1, 2, 3])
def test_destinations_that_are_copied(dim):
    import torch
    from paper_1009_2727_gb300.pic import Simulation
    w = W.parity_1d() if dim == 1 else W.shrink(W.parity_2d(), 48, 160) if dim == 2 else W.shrink3(W.parity_3d(), 24, 24, 64)
    sim = Simulation(w)
    sim.step(40)
    n = int(np.prod(sim.shape))
    for comp in (1, 3):
        want = sim.field(comp).reshape(-1)
        assert np.abs(want).max() > 0
        pinned = torch.zeros(n, dtype=torch.float64).pin_memory()
        odd = torch.zeros(2 * n + 1, dtype=torch.float32, device="cuda")
        for t, addr in ((pinned, pinned.data_ptr()), (odd, odd.data_ptr() + 4)):
            ptr = ctypes.cast(ctypes.c_void_p(addr), ctypes.POINTER(ctypes.c_double))
            assert sim.L.pic_get_field(sim.h, comp, ptr, 1) == 0
            torch.cuda.synchronize()
            got = t.numpy() if t is pinned else odd[1:].cpu().numpy().view(np.float64)
            assert np.array_equal(got, want)
    sim.close()
