"""Plasma rows that enter get their chunk's box from FP64 positions, their cells from the drifting frame's FP32 fraction:
at a cell's edge the two differ by a row. Such a chunk must not count as lying in its box (the window around the box
shows whether its electrons are in a field). The device functions compiled for the host, over many entry times."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include "pic_common.cuh"
using namespace picgb;
int main() {
  long seen = 0, differ = 0, wrong = 0;
  for (int ppc = 1; ppc <= 4; ppc *= 2)
    for (int e = 0; e < 400; e++) {
      const double dz = 1e-6 * (1.0 + 0.37 * e), h = dz / ppc, beta = std::sqrt(1.0 - 1.0 / (25.0 + e)), dt = dz / 299792458.0 * 0.7;
      for (int n = 1; n < 400; n++) {
        // the frame's shift of a step, and (even n) one within 1e-9 of a plasma row's offset in its cell
        double t = n * dt;
        if (n % 2 == 0) t = (n + (0.5 + n / 2 % ppc) / ppc + 1e-9 * ((n % 7) - 3)) * dz / (beta * kC);
        int sz;
        float fz;
        frame_of(beta * kC * t / dz, sz, fz);
        const long long m = (long long)std::ceil((200.0 * dz + beta * kC * t) / h - 0.5);   // the next row to enter
        for (long long r = m - 4 * ppc; r < m + 4 * ppc; r++) {
          const int row = (int)std::floor(((r + 0.5) * h - beta * kC * t) * (1.0 / dz));
          uint32_t cell;
          float ox, oz;
          lattice_site((int)r, 0, ppc, ppc, 0, 0, cell, ox, oz);
          const uint32_t k = z_key(cell_z(cell), oz);
          int z0, z1;
          key_rows(k, k, sz, fz, z0, z1);
          int fr;
          float tz;
          frame_z(cell, oz, sz, fz, fr, tz);
          seen++;
          differ += fr != row;
          wrong += z0 != fr || z1 != fr || key_rows_in(k, k, sz, fz, row, row) != (fr == row);
        }
      }
    }
  printf("%ld %ld %ld\n", seen, differ, wrong);
}
"""


def test_rows_outside_the_box(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    (tmp_path / "rows.cu").write_text(PROGRAM)
    subprocess.run([nvcc, "-std=c++17", "-Xcompiler", "-ffp-contract=off", "--expt-relaxed-constexpr", "-I",
                    os.path.join(ROOT, "paper_1009_2727_gb300", "csrc"), str(tmp_path / "rows.cu"), "-o",
                    str(tmp_path / "rows")], check=True)
    seen, differ, wrong = map(int, subprocess.run([str(tmp_path / "rows")], check=True, capture_output=True,
                                                  text=True).stdout.split())
    assert seen > 1_000_000 and differ > 0 and wrong == 0


def test_the_push_asks():
    """both the remembered and the scanned chunks pass the check before their box moves"""
    src = open(os.path.join(ROOT, "paper_1009_2727_gb300", "csrc", "pic_particles.cu")).read()
    body = src[src.index("bool chunk_at_rest("):src.index("void push_chunk(")]
    ask = body.index("!key_rows_in(lo, hi, pc.fr0_sz, pc.fr0_fz, ch.iz0, ch.iz1) || x0 < ch.ix0 || x1 > ch.ix1")
    assert body.index("if (!ch.rest)") < ask < body.index("o.rest = 1")
