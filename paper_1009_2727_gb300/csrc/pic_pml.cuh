// The split-field PML's update of one value, xi a + cf b with FP64 coefficients, rounded once to the fields' type.
#pragma once

namespace picgb {

// A coefficient as two FP32 values whose sum is it to 2^-48. One so small that its low part would underflow gets NaN:
// pml_step then takes the FP64 arithmetic for it.
inline void pml_pair(double v, float& hi, float& lo) {
  hi = (float)v;
  lo = (float)(v - (double)hi);
  if (v != 0.0 && v < 0x1p-100 && v > -0x1p-100) hi = lo = __builtin_nanf("");
}

// The products w.(x, y) a + w.(z, w) b as s + e, exact to 2^-44 of the terms' size m (four roundings of sums below 2^-22 m
// and the pairs' 2^-48): rounded 2^-43 m above (up) and below (dn).
__device__ __forceinline__ void pml_bounds(const float4& w, float a, float b, float& s, float& m, float& up, float& dn) {
  const float p = __fmul_rn(w.x, a), pe = __fmaf_rn(w.x, a, -p);
  const float r = __fmul_rn(w.z, b), re = __fmaf_rn(w.z, b, -r);
  s = __fadd_rn(p, r);
  const float v = __fadd_rn(s, -p);
  float e = __fadd_rn(__fadd_rn(p, -__fadd_rn(s, -v)), __fadd_rn(r, -v));
  e = __fadd_rn(e, __fadd_rn(pe, re));
  e = __fmaf_rn(w.y, a, e);
  e = __fmaf_rn(w.w, b, e);
  m = __fadd_rn(fabsf(p), fabsf(r));
  up = __fadd_rn(s, __fmaf_rn(m, 0x1p-43f, e));
  dn = __fadd_rn(s, __fmaf_rn(m, -0x1p-43f, e));
}

// x[q] a + f c[q] b (b negated: minus; f: E's c^2). FP64 instructions (conversions included) bounded the field kernels,
// since a warp's one occupies the SM for 16 cycles: the SMs with PML tiles were busy with them 70 to 90 % of the time. So
// FP32 fields take the coefficients as pairs t[q] = (x high, x low, f c high, f c low), and the products and the sum with
// their rounding errors. Where the bounds of the value round to the same FP32 value, the FP64 arithmetic rounds there too,
// and that is the result; else (one value in half a million without cancellation, more the more the terms cancel), and where
// a product overflows or is NaN, it is computed in FP64. Products so small that their rounding errors underflow are taken
// 2^64 times as large (ahead of a pulse its field falls through 1e-24 to zero within some tens of cells; in FP64 the tile
// there made Faraday 1.5 us longer, of 16 at 1536 x 224 nodes). The results are those of the FP64 arithmetic bit for bit
// down to the least normal number; below it (1e-38) they may differ by a unit of the last place.
template <class T>
__device__ __forceinline__ T pml_step(const double* x, const double* c, const float4* t, int q, double f, T a, T b,
                                      bool minus) {
  if (minus) b = -b;
  if constexpr (sizeof(T) == 4) {
    const float4 w = t[q];
    float s, m, up, dn;
    pml_bounds(w, a, b, s, m, up, dn);
    if (m >= 0x1p-80f) {
      if (up == dn) return up;
    } else {
      if (m == 0.0f && a == 0.0f && b == 0.0f) return s;   // no field: a zero of the products' sign
      pml_bounds(w, a * 0x1p64f, b * 0x1p64f, s, m, up, dn);
      if (up == dn) return up * 0x1p-64f;
    }
  }
  return T(x[q] * (double)a + f * c[q] * (double)b);
}

}  // namespace picgb
