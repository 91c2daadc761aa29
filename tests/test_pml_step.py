"""The FP32 fields' PML update (pairs of FP32 coefficients, FP64 where they cannot decide the rounding) against FP64
arithmetic rounded once, bit for bit (results below the least normal number: to a unit of the last place): coefficients over
the whole range of the tables, fields of any size, terms that cancel, fields whose rounding errors underflow, zeros of both
signs, infinities and NaN. Compiled for the host, where the rounding
of every operation is the device's."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r"""
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#define __device__
#define __forceinline__ inline
struct float4 { float x, y, z, w; };
static float __fmul_rn(float a, float b) { return a * b; }
static float __fadd_rn(float a, float b) { return a + b; }
static float __fmaf_rn(float a, float b, float c) { return std::fmaf(a, b, c); }
#include "pic_pml.cuh"
static uint64_t st;
static uint64_t rnd() {
  uint64_t z = (st += 0x9e3779b97f4a7c15ull);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}
static double uni() { return (rnd() >> 11) * 0x1p-53; }
static double sgn() { return rnd() & 1 ? 1.0 : -1.0; }
int main(int argc, char** argv) {
  const int mode = argv[1][0] - '0';
  const long n = 8000000;
  long bad = 0;
  st = 1234 + mode;
  for (long i = 0; i < n; i++) {
    // xi in [0, 1] down to 1e-40 (or the Cayley form's negative values), the coefficient about a time step, E's c^2
    double x = uni() < 0.2 ? std::pow(10.0, -40.0 * uni()) : uni();
    if (uni() < 0.1) x = -x;
    const double c = std::pow(10.0, -18.0 + 4.0 * uni()) * uni(), f = rnd() & 1 ? 1.0 : 299792458.0 * 299792458.0;
    const double big = mode == 0 ? std::pow(10.0, 14.0 * uni()) : mode == 1 ? std::pow(10.0, 20.0 * uni() - 8.0)
                     : mode == 2 ? std::pow(10.0, -46.0 + 26.0 * uni()) : std::pow(10.0, 84.0 * uni() - 45.0);
    float a = (float)(sgn() * big * uni());
    float b = (float)(sgn() * big * uni() / (f > 1.0 ? 3e8 : 1.0));
    if (mode == 1) b = (float)(-x * a / (f * c) * (1.0 + std::pow(2.0, -24.0 * uni()) * (uni() - 0.5)));   // terms that cancel
    if (mode == 3 && i % 16 == 0) a = (i & 16) ? 0.0f : -0.0f;
    if (mode == 3 && i % 24 == 0) b = (i & 8) ? 0.0f : -0.0f;
    if (mode == 3 && i % 1001 == 0) a = INFINITY;
    if (mode == 3 && i % 1003 == 0) b = -INFINITY;
    if (mode == 3 && i % 1007 == 0) b = NAN;
    float4 w;
    picgb::pml_pair(x, w.x, w.y);
    picgb::pml_pair(f * c, w.z, w.w);
    const bool minus = rnd() & 1;
    if (mode == 1 && minus) b = -b;
    const float got = picgb::pml_step<float>(&x, &c, &w, 0, f, a, b, minus);
    const float want = (float)(x * (double)a + f * c * (double)(minus ? -b : b));
    if (std::isnan(want) ? !std::isnan(got) : std::memcmp(&got, &want, 4) != 0)
      if (!(std::fabs(want) < 0x1p-126f && std::fabs((double)got - (double)want) <= 0x1p-149)) bad++;
  }
  printf("%ld\n", bad);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("pml")
    (d / "pml.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-ffp-contract=off", "-I",
                    os.path.join(ROOT, "paper_1009_2727_gb300", "csrc"), str(d / "pml.cpp"), "-o", str(d / "pml")], check=True)
    return str(d / "pml")


@pytest.mark.parametrize("mode", [0, 1, 2, 3], ids=["fields", "cancelling", "tiny", "everything"])
def test_bitwise_fp64(program, mode):
    out = subprocess.run([program, str(mode)], check=True, capture_output=True, text=True).stdout
    assert int(out) == 0
