// 1D path (z only; fields and positions depend on z, the three momentum
// components are kept) of the boosted-frame PIC step (Vay et al.,
// arXiv:1009.2727): the 2D/3D scheme with d/dx = d/dy = 0, which is Eq. 1db-1de
// of App. I for the transverse pair plus E_z from the longitudinal current.
//  - Faraday (the enlarged operator reduces to the Yee difference in 1D) with
//    Friedman's E_eff and the PML at both ends; Ampère with the PML;
//  - the composed filter along z (passes, compensation, stride or a set);
//  - gather (Yee locations or node-interpolated), Boris, 1D Esirkepov deposit;
//  - plasma rows through z_hi, ions fixed in the lab as a column current, a
//    current-sheet antenna, the lab-frame moving window.
// Layout: node k of every component at index k (arrays padded to 32 values);
// Ex, Ey, Bz, Jx, Jy at k, Ez, Bx, By, Jz at k + 1/2. Weights per unit area.
// A step is two launches: k1_fields (everything between two pushes, tile by tile in shared memory) and k1_push
// (electrons, ions, antenna). 1D grids are small: the step is bound by launches and latency, not by bandwidth.
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "pic_3d.h"
#include "pic_common.cuh"
#include "pic_dst.h"

namespace picgb {
namespace {

struct G1 {
  int nz;          // cells
  int n1p;         // padded node count of every array
  int lo, hi;      // particle domain [cells]
  double dz, idz, dt, z0;
};

inline unsigned nb1(long n, int b) { return (unsigned)((n + b - 1) / b); }

// valid range of component c (0..5: E then B; 6..8: J like E): half-staggered 0..nz-1, integer E 1..nz-1
// (tangential E vanishes on the PEC walls), integer B (Bz) 0..nz
__host__ __device__ inline bool half1(int c) {
  const int q = c >= 6 ? c - 6 : c;
  return q == 2 || q == 3 || q == 4;
}
__host__ __device__ inline void vr1(int c, int nz, int& lo, int& hi) {
  const int q = c >= 6 ? c - 6 : c;
  if (half1(q)) { lo = 0; hi = nz - 1; }
  else if (q < 3) { lo = 1; hi = nz - 1; }
  else { lo = 0; hi = nz; }
}

// B-spline shape of order 1 or 3 at offset s (cells)
template <class R>
__device__ __forceinline__ R shp(int order, R s) {
  const R a = fabs(s);
  if (order == 1) return a < R(1) ? R(1) - a : R(0);
  if (a < R(1)) return R(2) / R(3) - a * a + R(0.5) * a * a * a;
  if (a < R(2)) { const R t = R(2) - a; return t * t * t / R(6); }
  return R(0);
}

template <class T>
struct Pml1 {
  const T *sgI, *xiI, *cfI;   // integer positions
  const T *sgH, *xiH, *cfH;   // half positions
};

template <class T>
struct Taps1 {
  T c[2 * FILTER_HMAX + 1];
  int P, s;
};

// ---------------------------------------------------------------------------
// fields: one launch per step
//
// The step's order is Faraday, push, Ampère; between two pushes the fields need Ampère of one step, the moving
// window's shift, and Faraday, the Friedman history and the gather copies of the next. k1_fields does all of that for
// a tile of NT1 nodes in shared memory, recomputing what the tile's halo needs (the filters' reach), so that no
// grid-wide wait stands between the parts: it reads one set of the fields and writes the other. A step is then this
// kernel and k1_push. On these grids (a few hundred to a few thousand nodes) a launch costs more than its arithmetic:
// with one launch per part the fields of a step at 952 nodes (FP32, one pass on J) took 20 us of 52 us; this kernel
// takes 6.0 us, the step 12.7 us. It is bound by latency (load, four to six barriers), not by bytes.
constexpr int NT1 = 64;                              // nodes of a tile
constexpr int W1MAX = NT1 + 2 * FILTER_HMAX + 5;     // staged nodes: the gather filter's reach and one more each side
constexpr int JW1MAX = W1MAX + 2 * FILTER_HMAX;      // staged current: the current filter's reach on top
constexpr int FB1 = 384;                             // one thread per gather copy of the tile

// E, E^{n-1}, E-bar and B (three components of n1p nodes each)
template <class T>
struct Set1 {
  T *E, *Ep, *Eb, *B;
};

template <class T>
struct Fields1 {
  Set1<T> in, out;
  const T* J;      // the current deposited in the step that Ampère completes
  T* Jz;           // the next step's current, set to zero
  T *fE, *fB;      // gather copies
  T c1, c2, c3;    // E_eff = c1 E - c2 E^{n-1} + c3 E-bar
  T ha, hb;        // E-bar <- ha E + hb E-bar
  T dt, idz, c2idz, ie0;
  int ampere, faraday;             // the parts to run
  int filt_j, filt_g, nodal;       // current filter, gather filter, node-interpolated gather copies
  int shift, H;                    // window shift (cells) between the parts; reach of a filter that is on
};

template <class T>
__global__ void __launch_bounds__(FB1) k1_fields(G1 g, Pml1<T> pm, Taps1<T> t, Fields1<T> a) {
  __shared__ T sJ[3][JW1MAX];
  __shared__ T sE[3][W1MAX], sEp[3][W1MAX], sEb[3][W1MAX], sB[3][W1MAX], sV[3][W1MAX];
  __shared__ T sP[9][W1MAX];   // PML tables: sigma, xi, coefficient at integer and half nodes (Ampère), half nodes (Faraday)
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  const int n = g.n1p, nz = g.nz, H = a.H, sh = a.shift;
  const int t0 = blockIdx.x * NT1;
  const int W = NT1 + 2 * H + 5, JW = W + 2 * H;
  // staged node i is node p0 + i before the shift and p0 + i - sh after it; staged current j is node p0 - H + j
  const int p0 = t0 - H - 3 + sh;
  if (a.ampere) {
    for (int e = threadIdx.x; e < 3 * JW; e += FB1) {
      const int q = e / JW, i = e - q * JW, k = p0 - H + i;
      sJ[q][i] = (k >= 0 && k <= nz) ? a.J[q * n + k] : T(0);
    }
  }
  for (int e = threadIdx.x; e < 3 * W; e += FB1) {
    const int q = e / W, i = e - q * W, k = p0 + i;
    const bool in = k >= 0 && k <= nz;
    sE[q][i] = in ? a.in.E[q * n + k] : T(0);
    sB[q][i] = in ? a.in.B[q * n + k] : T(0);
    sEp[q][i] = in ? a.in.Ep[q * n + k] : T(0);
    sEb[q][i] = in ? a.in.Eb[q * n + k] : T(0);
  }
  for (int e = threadIdx.x; e < 9 * W; e += FB1) {
    const int q = e / W, i = e - q * W, k = p0 + i - (q >= 6 ? sh : 0);
    const T* tab = q == 0 ? pm.sgI : q == 1 ? pm.xiI : q == 2 ? pm.cfI : q % 3 == 0 ? pm.sgH : q % 3 == 1 ? pm.xiH : pm.cfH;
    if (k >= 0 && k <= nz) sP[q][i] = tab[k];
  }
  __syncthreads();
  if (a.ampere) {
    // Ampère with the PML: Ex(k) += dt (-c^2 dBy/dz - Jx/eps0), Ey(k) += dt (c^2 dBx/dz - Jy/eps0),
    // Ez(k+1/2) += -dt Jz/eps0; no current in the PML, where the curl term is damped. Every node reads its own E and
    // the unchanged B only, so E is updated in place.
    for (int e = threadIdx.x; e < 3 * W; e += FB1) {
      const int q = e / W, i = e - q * W, k = p0 + i;
      int lo, hi;
      vr1(q, nz, lo, hi);
      if (k < lo || k > hi || i < 1) continue;
      T d = T(0);
      if (q == 0) d = -a.c2idz * (sB[1][i] - sB[1][i - 1]);
      if (q == 1) d = a.c2idz * (sB[0][i] - sB[0][i - 1]);
      const int pt = q == 2 ? 3 : 0;
      const T old = sE[q][i];
      if (sP[pt][i] > T(0)) {
        sE[q][i] = sP[pt + 1][i] * old + sP[pt + 2][i] * d;
      } else {
        T j;
        if (a.filt_j) {
          j = T(0);
          const T* c = sJ[q] + i + H - t.P * t.s;   // staged values off the grid are zero
          for (int m = 0; m <= 2 * t.P; m++) j += t.c[m] * c[m * t.s];
        } else {
          j = sJ[q][i + H];
        }
        sE[q][i] = old + a.dt * (d - j * a.ie0);
      }
    }
    __syncthreads();
  }
  if (sh > 0) {
    // the window's shift: node k of every array takes the value of node k + sh, on the component's valid range
    for (int e = threadIdx.x; e < 3 * W; e += FB1) {
      const int q = e / W, i = e - q * W, k = p0 + i - sh;
      int lo, hi;
      vr1(q, nz, lo, hi);
      if (k < lo || k > hi) { sE[q][i] = T(0); sEp[q][i] = T(0); sEb[q][i] = T(0); }
      vr1(3 + q, nz, lo, hi);
      if (k < lo || k > hi) sB[q][i] = T(0);
    }
    __syncthreads();
  }
  const int k0 = p0 - sh;   // node of staged index 0 from here on
  if (!a.faraday) {
    for (int e = threadIdx.x; e < 3 * NT1; e += FB1) {
      const int q = e / NT1, i = e - q * NT1 + t0 - k0, k = k0 + i;
      if (k > nz) continue;
      a.out.E[q * n + k] = sE[q][i];
      a.out.Ep[q * n + k] = sEp[q][i];
      a.out.Eb[q * n + k] = sEb[q][i];
      a.out.B[q * n + k] = sB[q][i];
      a.Jz[q * n + k] = T(0);
    }
    return;
  }
  // Faraday with E_eff and the PML: Bx(k+1/2) += dt dEy/dz, By(k+1/2) -= dt dEx/dz, and the average of the old and
  // the new B for the gather, on the tile and the filter's reach (staged indices 1 .. W - 2); the tile's own nodes
  // are written with the Friedman history E-bar <- ha E + hb E-bar, E^{n-1} <- E
  for (int e = threadIdx.x; e < 3 * W; e += FB1) {
    const int q = e / W, i = e - q * W, k = k0 + i;
    const bool in = k >= 0 && k <= nz;
    const T old = sB[q][i];
    T nw = old;
    if (in && q < 2 && k <= nz - 1 && i + 1 < W) {
      const int ce = q == 0 ? 1 : 0;
      const T e1 = a.c1 * sE[ce][i + 1] - a.c2 * sEp[ce][i + 1] + a.c3 * sEb[ce][i + 1];
      const T e0 = a.c1 * sE[ce][i] - a.c2 * sEp[ce][i] + a.c3 * sEb[ce][i];
      const T d = (q == 0 ? T(1) : T(-1)) * (e1 - e0) * a.idz;
      nw = sP[6][i] > T(0) ? sP[7][i] * old + sP[8][i] * d : old + a.dt * d;
    }
    sV[q][i] = in ? T(0.5) * (old + nw) : T(0);
    if (in && k >= t0 && k < t0 + NT1) {
      const T ev = sE[q][i];
      a.out.B[q * n + k] = nw;
      a.out.E[q * n + k] = ev;
      a.out.Ep[q * n + k] = ev;
      a.out.Eb[q * n + k] = a.ha * ev + a.hb * sEb[q][i];
      a.Jz[q * n + k] = T(0);
    }
  }
  __syncthreads();
  // gather copies: the composed filter along z of E and of the averaged B (zero off the component's valid range), or
  // the values themselves; for the 'momentum conserving' gather (Sec. 5) a half-staggered component (Ez, Bx, By)
  // becomes the mean of its two nearest values (off the grid: zero)
  for (int e = threadIdx.x; e < 6 * NT1; e += FB1) {
    const int c = e / NT1, k = t0 + e - c * NT1, i = k - k0;
    if (k > nz) continue;
    const T* F = c < 3 ? sE[c] : sV[c - 3];
    int lo, hi;
    vr1(c, nz, lo, hi);
    auto copy_at = [&](int kk, int ii) {
      if (!a.filt_g) return F[ii];
      T acc = T(0);
      if (kk >= lo && kk <= hi) {
        const T* w = F + ii - t.P * t.s;   // staged values off the grid are zero
        for (int m = 0; m <= 2 * t.P; m++) acc += t.c[m] * w[m * t.s];
      }
      return acc;
    };
    T v = copy_at(k, i);
    if (a.nodal && half1(c)) v = T(0.5) * ((k >= 1 ? copy_at(k - 1, i - 1) : T(0)) + v);
    (c < 3 ? a.fE + c * n : a.fB + (c - 3) * n)[k] = v;
  }
}

// ---------------------------------------------------------------------------
// particles
template <class T>
struct Parts1 {
  double* z;
  T *ux, *uy, *uz, *w;
  uint32_t* id;
};

struct Ctrl1 {
  int count;
  int status;
};

// plasma rows [m0, m0 + nrow): row m at z' = (m + 1/2) h - beta c t, density gamma n0(gamma (m + 1/2) h),
// weight n' dz / ppc_z per unit area; rows without plasma, or below z_lo, are stored dead (w = 0)
struct Lat1 {
  double h, gamma, beta, n0, z_start_lab, ramp_lab, length_lab, dz;
  int ppc;
};

__host__ __device__ inline double lab_density1(const Lat1& L, double zl) {
  if (zl < L.z_start_lab) return 0.0;
  const double r = zl - L.z_start_lab;
  if (L.ramp_lab > 0.0 && r < L.ramp_lab) return L.n0 * r / L.ramp_lab;
  const double plateau_end = L.ramp_lab + L.length_lab;
  if (L.length_lab > 0.0 && r >= plateau_end) return 0.0;
  return L.n0;
}

// rows waiting to be stored in the slots at .. at + nrow - 1
struct Rows1 {
  long long m0;
  int nrow, at;
  double t, zlo;
};

// state of lattice row m entering at time t
template <class T>
__device__ __forceinline__ void row_state(const Lat1& L, long long m, double t, double zlo, double& z, T& uz, T& w) {
  const double zlat = (m + 0.5) * L.h;
  const double n = L.gamma * lab_density1(L, L.gamma * zlat);
  z = zlat - L.beta * kC * t;
  uz = T(-L.gamma * L.beta * kC);
  w = (n > 0.0 && z >= zlo) ? T(n * L.dz / (double)L.ppc) : T(0);
}

template <class T>
__global__ void k1_inject(Parts1<T> p, Ctrl1* ctrl, Lat1 L, Rows1 r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= r.nrow) return;
  const int q = r.at + i;
  double z;
  T uz, w;
  row_state<T>(L, r.m0 + i, r.t, r.zlo, z, uz, w);
  p.z[q] = z;
  p.ux[q] = T(0);
  p.uy[q] = T(0);
  p.uz[q] = uz;
  p.w[q] = w;
  p.id[q] = (uint32_t)(r.m0 + i);
  if (i == 0) ctrl->count = r.at + r.nrow;
}

// current-sheet antenna: J_y(k) += K w_k / dz over eight nodes from k0
struct Ant1 {
  int k0, on;
  double v[8];
};

// the rigid ions' rows of one step (off: on = 0)
struct Ions1 {
  long long mlo, mhi;
  double t0, t1;
  int on;
};

// share of a row's shape samples on the nodes <= k (the 1D Esirkepov flux of a row at Z, in cells, through the face
// above node k), in closed form from the four (two) weights
template <int ORD>
__device__ __forceinline__ double cum_shape1(double Z, int k) {
  const double f = floor(Z), t = Z - f;
  const int j = k - ((int)f - (ORD == 3 ? 1 : 0));   // node k in the row's stencil
  if (j < 0) return 0.0;
  if (ORD == 3) {
    if (j >= 3) return 1.0;
    const double t2 = t * t, t3 = t2 * t, s = 1.0 - t;
    const double w0 = s * s * s * (1.0 / 6.0);
    if (j == 0) return w0;
    if (j == 1) return w0 + (2.0 / 3.0 - t2 + 0.5 * t3);
    return 1.0 - t3 * (1.0 / 6.0);
  }
  return j >= 1 ? 1.0 : 1.0 - t;
}

// One electron per thread: gather -> Boris -> move -> 1D Esirkepov; removal after the deposit when it leaves
// [z_lo, z_hi + dz). The rows that entered at the end of the last step are created in their slots here. The blocks past
// the electrons' add the rigid ions' column current, a warp per node with its lanes over the rows: one thread per
// node with generic shape sums took 150 us a step in FP64 at 400 nodes and 4 rows a cell. Block 0 adds the antenna.
// Bound by the latency of one particle's chain (FP32: 10.6 us at 9100 electrons in 24,000 slots, 26.5 us with generic
// shape functions and lanes of one cell on the same words) and, in FP64, by the FP64 pipe (17 us with the ions at 2500
// electrons and 400 nodes; 203 us before).
// A block takes PB1 consecutive slots (injected row by row, so close in z) and sums their current in a shared window
// over its cells, then adds the window to J; a block spread wider than the window adds to J directly. Thread t takes
// slot (9 t) mod PB1 of the block: neighbouring lanes then sit about a cell apart, where consecutive slots of one
// cell would meet on every shared atomic (FP32 and FP64 shared adds retry on a collision).
// Threads of a block: the FP64 pipe of an SM serves two lanes a cycle, so FP64 blocks are small and spread over the SMs
// (2500 electrons, 400 nodes: 17 us in blocks of 64, 24 us in blocks of 256; FP32 11.2 us in blocks of 256, 10.6 in
// blocks of 128).
template <class T>
constexpr int push_threads1() { return sizeof(T) == 8 ? 64 : 128; }
constexpr int JW1 = 192;

template <class T, int ORD, bool MC>
__global__ void __launch_bounds__(push_threads1<T>()) k1_push(G1 g, const T* fE, const T* fB, T* J,
                                               Parts1<T> p, int count, Ctrl1* ctrl, T kq, T qe, double zlo,
                                               double zhi1, Lat1 L, Rows1 rows, Ions1 ions, Ant1 ant, int nbp) {
  constexpr int NG = ORD + 1, ND = NG + 1, OFF = ORD == 3 ? 1 : 0, PB1 = push_threads1<T>();
  static_assert((PB1 & (PB1 - 1)) == 0, "(9 t) mod PB1 visits every slot once");
  const int n = g.n1p;
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  if ((int)blockIdx.x >= nbp) {
    // ions fixed in the lab (PR-9): J_z(k+1/2) += -(e/dt) sum over the live rows of w_m (C(Z1, k) - C(Z0, k))
    const int k = ((int)blockIdx.x - nbp) * (PB1 / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (k > g.nz) return;   // warp-uniform
    const double vsh = L.beta * kC;
    long long m0 = (long long)floor(((k - 4) * g.dz + g.z0 + vsh * ions.t0) / L.h - 0.5);
    long long m1 = (long long)ceil(((k + 4) * g.dz + g.z0 + vsh * ions.t0) / L.h - 0.5);
    if (m0 < ions.mlo) m0 = ions.mlo;
    if (m1 > ions.mhi - 1) m1 = ions.mhi - 1;
    double acc = 0.0;
    for (long long m = m0 + lane; m <= m1; m += 32) {
      const double zl = (m + 0.5) * L.h;
      const double nd = L.gamma * lab_density1(L, L.gamma * zl);
      if (nd <= 0.0) continue;
      const double w = nd * L.dz / (double)L.ppc;
      const double Z0 = (zl - vsh * ions.t0 - g.z0) * g.idz, Z1 = (zl - vsh * ions.t1 - g.z0) * g.idz;
      acc += w * (cum_shape1<ORD>(Z1, k) - cum_shape1<ORD>(Z0, k));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_down_sync(0xffffffffu, acc, o);
    if (lane == 0 && acc != 0.0) atomicAdd(J + 2 * n + k, T(-kQe / g.dt * acc));
    return;
  }
  __shared__ T sJ[3][JW1];
  __shared__ int s_lo, s_hi;
  if (threadIdx.x == 0) { s_lo = INT_MAX; s_hi = INT_MIN; }
  for (int e = threadIdx.x; e < 3 * JW1; e += PB1) (&sJ[0][0])[e] = T(0);
  const int j = blockIdx.x * PB1 + ((9 * threadIdx.x) & (PB1 - 1));
  T w = T(0), u0 = T(0), u1 = T(0), u2 = T(0);
  double z = 0.0;
  if (j < count) {
    const int r = j - rows.at;
    if (rows.nrow > 0 && r >= 0 && r < rows.nrow) {
      row_state<T>(L, rows.m0 + r, rows.t, rows.zlo, z, u2, w);
      p.id[j] = (uint32_t)(rows.m0 + r);
      p.w[j] = w;
      if (w == T(0)) {   // a dead slot is stored whole; a live one is stored below
        p.z[j] = z; p.ux[j] = T(0); p.uy[j] = T(0); p.uz[j] = u2;
      }
    } else {
      w = p.w[j];
      if (w > T(0)) { z = p.z[j]; u0 = p.ux[j]; u1 = p.uy[j]; u2 = p.uz[j]; }
    }
  }
  if (blockIdx.x == 0) {
    if (threadIdx.x == 0 && rows.nrow > 0) ctrl->count = count;
    if (ant.on && threadIdx.x < 8) {
      const int k = ant.k0 + (int)threadIdx.x;
      if (k >= 0 && k <= g.nz && ant.v[threadIdx.x] != 0.0) atomicAdd(J + n + k, T(ant.v[threadIdx.x]));
    }
  }
  const bool live = w > T(0);
  double Z = 0.0;
  int f = 0;
  if (live) {
    Z = (z - g.z0) * g.idz;
    f = (int)floor(Z);
  }
  const int flo = __reduce_min_sync(0xffffffffu, live ? f : INT_MAX);
  const int fhi = __reduce_max_sync(0xffffffffu, live ? f : INT_MIN);
  __syncthreads();
  if ((threadIdx.x & 31) == 0 && flo <= fhi) { atomicMin(&s_lo, flo); atomicMax(&s_hi, fhi); }
  __syncthreads();
  if (s_hi < s_lo) return;   // block-uniform: no live electron here
  // the deposit of a particle in cell f (moving less than a cell) touches nodes f - 2 .. f + 3
  const int base = s_lo - 2, span = s_hi - s_lo + 6;
  const bool win = span <= JW1;
  if (live) {
    // shape weights from the fractional offset: integer nodes from f - OFF, half-staggered ones from fh - OFF
    const T ti = T(Z - f);
    const int fh = ti >= T(0.5) ? f : f - 1;
    const T th = ti >= T(0.5) ? ti - T(0.5) : ti + T(0.5);
    T wi[NG], wh[NG];
    if constexpr (ORD == 3) { weights3<T>(ti, wi); weights3<T>(th, wh); }
    else { weights1<T>(ti, wi); weights1<T>(th, wh); }
    T EB[6];
    const bool inside = f - OFF - 1 >= 0 && f + NG <= g.nz;
#pragma unroll
    for (int c = 0; c < 6; c++) {
      const T* F = c < 3 ? fE + c * n : fB + (c - 3) * n;
      const bool hf = !MC && half1(c);
      const int k0 = (hf ? fh : f) - OFF;
      T acc = T(0);
#pragma unroll
      for (int b = 0; b < NG; b++)
        if (inside || (k0 + b >= 0 && k0 + b <= g.nz)) acc += F[k0 + b] * (hf ? wh[b] : wi[b]);
      EB[c] = acc;
    }
    // relativistic Boris push (textbook), one division each for k / gamma and 2 / (1 + t^2)
    const T ic2 = T(1.0 / (kC * kC));
    const T um0 = u0 + kq * EB[0], um1 = u1 + kq * EB[1], um2 = u2 + kq * EB[2];
    const T kg = kq / sqrt(T(1) + (um0 * um0 + um1 * um1 + um2 * um2) * ic2);
    const T t0 = kg * EB[3], t1 = kg * EB[4], t2 = kg * EB[5];
    const T sf = T(2) / (T(1) + (t0 * t0 + t1 * t1 + t2 * t2));
    const T s0 = sf * t0, s1 = sf * t1, s2 = sf * t2;
    const T up0 = um0 + (um1 * t2 - um2 * t1), up1 = um1 + (um2 * t0 - um0 * t2), up2 = um2 + (um0 * t1 - um1 * t0);
    const T pl0 = um0 + (up1 * s2 - up2 * s1), pl1 = um1 + (up2 * s0 - up0 * s2), pl2 = um2 + (up0 * s1 - up1 * s0);
    u0 = pl0 + kq * EB[0]; u1 = pl1 + kq * EB[1]; u2 = pl2 + kq * EB[2];
    const T ig = T(1) / sqrt(T(1) + (u0 * u0 + u1 * u1 + u2 * u2) * ic2);
    const double zn = z + g.dt * (double)(u2 * ig);
    const double Zn = (zn - g.z0) * g.idz;
    p.z[j] = zn;
    p.ux[j] = u0; p.uy[j] = u1; p.uz[j] = u2;
    if (zn < zlo || zn >= zhi1) p.w[j] = T(0);
    // 1D Esirkepov: Jz(k+1/2) = -(q w/dt) sum_{k' <= k} (S1 - S0)(k'); Jx, Jy = q w v (S0 + S1)/(2 dz)
    const int fn = (int)floor(Zn);
    const int b0 = (f < fn ? f : fn) - OFF;
    T wn[NG];
    const T tn = T(Zn - fn);
    if constexpr (ORD == 3) weights3<T>(tn, wn);
    else weights1<T>(tn, wn);
    const T qw = qe * w;
    const T cz = -qw / T(g.dt), ct = qw * T(0.5) * T(g.idz);
    const T cx = ct * (u0 * ig), cy = ct * (u1 * ig);
    const bool o0 = f - OFF > b0, o1 = fn - OFF > b0;
    T run = T(0);
#pragma unroll
    for (int a = 0; a < ND; a++) {
      // a stencil starts at b0 or one node above
      const T S0 = o0 ? (a >= 1 ? wi[a - 1] : T(0)) : (a < NG ? wi[a] : T(0));
      const T S1 = o1 ? (a >= 1 ? wn[a - 1] : T(0)) : (a < NG ? wn[a] : T(0));
      run += S1 - S0;
      const int k = b0 + a;
      if (k < 0 || k > g.nz) continue;
      const T ss = S0 + S1;
      const T jz = a < ND - 1 ? cz * run : T(0), jx = cx * ss, jy = cy * ss;
      const int l = k - base;
      if (win && l >= 0 && l < span) {
        if (jz != T(0)) atomicAdd(&sJ[2][l], jz);
        if (jx != T(0)) atomicAdd(&sJ[0][l], jx);
        if (jy != T(0)) atomicAdd(&sJ[1][l], jy);
      } else {
        if (jz != T(0)) atomicAdd(J + 2 * n + k, jz);
        if (jx != T(0)) atomicAdd(J + k, jx);
        if (jy != T(0)) atomicAdd(J + n + k, jy);
      }
    }
  }
  __syncthreads();
  if (win) {
    for (int e = threadIdx.x; e < 3 * span; e += PB1) {
      const int q = e / span, l = e - q * span, k = base + l;
      const T v = sJ[q][l];
      if (v != T(0) && k >= 0 && k <= g.nz) atomicAdd(J + q * n + k, v);
    }
  }
}

// charge density: electrons and the ion rows at time t
template <class T>
__global__ void k1_rho_e(G1 g, Parts1<T> p, const Ctrl1* ctrl, int order, double* rho) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= ctrl->count) return;
  const double w = (double)p.w[j];
  if (!(w > 0.0)) return;
  const double Z = (p.z[j] - g.z0) * g.idz;
  const int f = (int)floor(Z);
  for (int k = f - 3; k <= f + 3; k++) {
    if (k < 0 || k > g.nz) continue;
    const double s = shp<double>(order, Z - k);
    if (s != 0.0) atomicAdd(rho + k, -kQe * w * s * g.idz);
  }
}

__global__ void k1_rho_i(G1 g, Lat1 L, int order, long long mlo, long long mhi, double t, double* rho) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k > g.nz) return;
  const double vsh = L.beta * kC;
  long long m0 = (long long)floor(((k - 3) * g.dz + g.z0 + vsh * t) / L.h - 0.5);
  long long m1 = (long long)ceil(((k + 3) * g.dz + g.z0 + vsh * t) / L.h - 0.5);
  if (m0 < mlo) m0 = mlo;
  if (m1 > mhi - 1) m1 = mhi - 1;
  double acc = 0.0;
  for (long long m = m0; m <= m1; m++) {
    const double zl = (m + 0.5) * L.h;
    const double n = L.gamma * lab_density1(L, L.gamma * zl);
    if (n <= 0.0) continue;
    acc += n * L.dz / (double)L.ppc * shp<double>(order, (zl - vsh * t - g.z0) * g.idz - k);
  }
  rho[k] += kQe * acc * g.idz;
}

// diagnostics: [0] live electrons, [1] field energy per unit area, [2] weight above the lab gamma threshold
template <class T>
__global__ void __launch_bounds__(256) k1_stats(G1 g, const T* E, const T* B, Parts1<T> p, const Ctrl1* ctrl,
                                                double gam, double be, double trap, double* out) {
  __shared__ double red[3][256];
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nthr = gridDim.x * blockDim.x;
  double ne = 0, en = 0, wt = 0;
  for (int j = tid; j < ctrl->count; j += nthr) {
    const double w = (double)p.w[j];
    if (!(w > 0.0)) continue;
    ne += 1.0;
    if (trap > 0.0) {
      const double ux = p.ux[j], uy = p.uy[j], uz = p.uz[j];
      const double gp = sqrt(1.0 + (ux * ux + uy * uy + uz * uz) / (kC * kC));
      if (gam * (gp + be * uz / kC) > trap) wt += w;
    }
  }
  const int n = g.n1p;
  for (int k = tid; k <= g.nz; k += nthr) {
    double e2 = 0, b2 = 0;
    for (int c = 0; c < 3; c++) {
      const double ev = E[c * n + k], bv = B[c * n + k];
      e2 += ev * ev; b2 += bv * bv;
    }
    en += 0.5 * (kEps0 * e2 + b2 * (kEps0 * kC * kC)) * g.dz;
  }
  red[0][threadIdx.x] = ne; red[1][threadIdx.x] = en; red[2][threadIdx.x] = wt;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o)
      for (int c = 0; c < 3; c++) red[c][threadIdx.x] += red[c][threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0)
    for (int c = 0; c < 3; c++) atomicAdd(out + c, red[c][0]);
}

// compaction of the live electrons into the other buffer set (order kept)
template <class T>
__global__ void k1_live_per_block(Parts1<T> p, const Ctrl1* ctrl, int* bc) {
  __shared__ int s;
  if (threadIdx.x == 0) s = 0;
  __syncthreads();
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int live = (j < ctrl->count && p.w[j] > T(0)) ? 1 : 0;
  const int wsum = __popc(__ballot_sync(0xffffffffu, live));
  if ((threadIdx.x & 31) == 0 && wsum) atomicAdd(&s, wsum);
  __syncthreads();
  if (threadIdx.x == 0) bc[blockIdx.x] = s;
}

__global__ void __launch_bounds__(1024) k1_scan_blocks(int* bc, int nb, Ctrl1* ctrl) {
  __shared__ int part[1024];
  const int per = (nb + 1023) / 1024;
  const int b0 = threadIdx.x * per, b1 = min(nb, b0 + per);
  int s = 0;
  for (int b = b0; b < b1; b++) s += bc[b];
  part[threadIdx.x] = s;
  __syncthreads();
  for (int o = 1; o < 1024; o <<= 1) {
    const int v = threadIdx.x >= o ? part[threadIdx.x - o] : 0;
    __syncthreads();
    part[threadIdx.x] += v;
    __syncthreads();
  }
  int run = part[threadIdx.x] - s;
  for (int b = b0; b < b1; b++) {
    const int c = bc[b];
    bc[b] = run;
    run += c;
  }
  if (threadIdx.x == 1023) ctrl->count = part[1023];
}

template <class T>
__global__ void k1_scatter(Parts1<T> src, Parts1<T> dst, const int* bo, int n_old) {
  __shared__ int wo[8];
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  const int live = (j < n_old && src.w[j] > T(0)) ? 1 : 0;
  const unsigned m = __ballot_sync(0xffffffffu, live);
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (lane == 0) wo[wid] = __popc(m);
  __syncthreads();
  if (!live) return;
  int off = bo[blockIdx.x];
  for (int q = 0; q < wid; q++) off += wo[q];
  const int d = off + __popc(m & ((1u << lane) - 1u));
  dst.z[d] = src.z[j]; dst.ux[d] = src.ux[j]; dst.uy[d] = src.uy[j]; dst.uz[d] = src.uz[j];
  dst.w[d] = src.w[j]; dst.id[d] = src.id[j];
}

template <class T>
__global__ void k1_out(int n, const T* F, double* out) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) out[k] = (double)F[k];
}
template <class T>
__global__ void k1_in(int n, const double* in, T* F) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) F[k] = T(in[k]);
}

// ---------------------------------------------------------------------------
template <class T>
class Sim1 : public Sim3Api {
 public:
  Sim1(const pic_config& c, pic_alloc_fn a, pic_free_fn f, void* u, cudaStream_t s_)
      : cfg(c), alloc(a), freef(f), user(u), s(s_) {}
  ~Sim1() override {
    cudaStreamSynchronize(s);
    for (auto& p : allocs) {
      if (freef) freef(p.first, p.second, (void*)s, user);
      else cudaFree(p.first);
    }
    for (auto e : tev) cudaEventDestroy(e);
    if (ev0) cudaEventDestroy(ev0);
    if (ev1) cudaEventDestroy(ev1);
  }

  int fail(int code, const char* msg) {
    if (st == PIC_OK) { st = code; err = msg; }
    return code;
  }

  template <class U>
  U* dal(size_t n) {
    size_t bytes = std::max<size_t>(n * sizeof(U), 16);
    bytes = (bytes + 255) & ~size_t(255);
    void* p = nullptr;
    if (alloc) p = alloc(bytes, (void*)s, user);
    else if (cudaMalloc(&p, bytes) != cudaSuccess) p = nullptr;
    if (!p) return nullptr;
    allocs.push_back({p, bytes});
    cudaMemsetAsync(p, 0, bytes, s);
    return (U*)p;
  }

  int init() {
    const pic_config* c = &cfg;
    if (c->nz < 16 || !(c->dz_lab > 0)) return fail(PIC_EINVAL, "1D: nz >= 16 and dz_lab > 0");
    gamma = c->gamma_boost < 1.0 ? 1.0 : c->gamma_boost;
    beta = std::sqrt(1.0 - 1.0 / (gamma * gamma));
    g.nz = c->nz;
    g.n1p = ((c->nz + 1 + 31) / 32) * 32;
    g.dz = (1.0 + beta) * gamma * c->dz_lab;          // Sec. 5.1.1
    g.idz = 1.0 / g.dz;
    g.z0 = 0.0;
    const double th = c->theta;
    const double lim = g.dz / kC * std::sqrt((2.0 + th) / (2.0 + 3.0 * th));
    g.dt = c->dt > 0.0 ? c->dt : c->courant * lim;
    if (!(g.dt > 0.0)) return fail(PIC_EINVAL, "dt <= 0");
    if (g.dt > lim * (1.0 + 1e-12)) return fail(PIC_ECFL, "dt above the 1D stability limit");
    if (c->moving_window && gamma > 1.0) return fail(PIC_EINVAL, "1D moving window: lab frame only");
    FilterSpec fs{};
    fs.passes = c->filter_passes; fs.stride = c->filter_stride; fs.compensate = c->filter_compensate;
    for (int q = 0; q < 4; q++) fs.strides[q] = c->filter_stride_set[q];
    const int H = filter_halo(fs);
    P = c->filter_passes + (c->filter_compensate ? 1 : 0);
    const int guard = c->particle_guard >= 0 ? c->particle_guard : (c->shape_order == 3 ? 3 : 2) + H + 2;
    if (guard < (c->shape_order == 3 ? 3 : 2) + H + 1) return fail(PIC_EINVAL, "particle guard too small");
    g.lo = c->pml_cells + guard;
    g.hi = c->nz - c->pml_cells - guard;
    if (g.hi - g.lo < 2 || g.lo < 4) return fail(PIC_EINVAL, "1D box too small for the PML and guard");
    // composed taps (dense over the halo for a wide-band filter)
    const bool wide = fs.strides[0] > 0;
    const int R = wide ? H : P;
    std::vector<double> t(2 * R + 1, 0.0);
    t[R] = 1.0;
    for (int q = 0; q < (wide ? 4 : 1); q++) {
      const int stq = wide ? fs.strides[q] : 1;
      if (stq <= 0) break;
      for (int pp = 0; pp < P; pp++) {
        const double al = pp < c->filter_passes ? 0.5 : 0.5 * c->filter_passes + 1.0;
        std::vector<double> o(2 * R + 1, 0.0);
        for (int m = 0; m <= 2 * R; m++) {
          o[m] += al * t[m];
          if (m - stq >= 0) o[m] += 0.5 * (1.0 - al) * t[m - stq];
          if (m + stq <= 2 * R) o[m] += 0.5 * (1.0 - al) * t[m + stq];
        }
        t = o;
      }
    }
    for (int m = 0; m < 2 * FILTER_HMAX + 1; m++) taps.c[m] = m <= 2 * R ? T(t[m]) : T(0);
    taps.P = R;
    taps.s = wide ? 1 : c->filter_stride;
    nodal = c->gather_scheme == 1;
    const int n = g.n1p;
    // two sets of the fields and of the current: k1_fields reads one and writes the other
    for (int q = 0; q < 2; q++) {
      fs2[q].E = dal<T>(3 * n); fs2[q].Ep = dal<T>(3 * n); fs2[q].Eb = dal<T>(3 * n); fs2[q].B = dal<T>(3 * n);
      J2[q] = dal<T>(3 * n);
      if (!fs2[q].E || !fs2[q].Ep || !fs2[q].Eb || !fs2[q].B || !J2[q]) return fail(PIC_ENOMEM, "allocation failed");
    }
    fE = dal<T>(3 * n); fB = dal<T>(3 * n);
    rho = dal<double>(n); outd = dal<double>(n); sred = dal<double>(4); ctrl = dal<Ctrl1>(1);
    if (!fE || !fB || !rho || !outd || !sred || !ctrl) return fail(PIC_ENOMEM, "allocation failed");
    // PML tables at integer and half positions
    std::vector<T> sg(2 * n, T(0)), xi(2 * n, T(1)), cf(2 * n, T(g.dt));
    for (int h = 0; h < 2; h++)
      for (int k = 0; k <= c->nz; k++) {
        const double pos = k + 0.5 * h;
        double sgv = 0.0;
        const int L = c->pml_cells;
        if (L > 0) {
          double d = 0.0;
          if (pos < L) d = L - pos;
          if (pos > c->nz - L) d = pos - (c->nz - L);
          if (d > 0.0) sgv = c->pml_sigma_max * kC / g.dz * std::pow(d / c->pml_delta, c->pml_power);
        }
        const double x = c->pml_xi_exp ? std::exp(-sgv * g.dt) : (1.0 - 0.5 * sgv * g.dt) / (1.0 + 0.5 * sgv * g.dt);
        sg[h * n + k] = T(sgv);
        xi[h * n + k] = T(x);
        cf[h * n + k] = T(sgv > 0.0 ? (1.0 - x) / sgv : g.dt);
      }
    T* dsg = dal<T>(2 * n);
    T* dxi = dal<T>(2 * n);
    T* dcf = dal<T>(2 * n);
    if (!dsg || !dxi || !dcf) return fail(PIC_ENOMEM, "allocation failed");
    cudaMemcpyAsync(dsg, sg.data(), sizeof(T) * 2 * n, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dxi, xi.data(), sizeof(T) * 2 * n, cudaMemcpyHostToDevice, s);
    cudaMemcpyAsync(dcf, cf.data(), sizeof(T) * 2 * n, cudaMemcpyHostToDevice, s);
    cudaStreamSynchronize(s);
    pm.sgI = dsg; pm.xiI = dxi; pm.cfI = dcf;
    pm.sgH = dsg + n; pm.xiH = dxi + n; pm.cfH = dcf + n;
    return cudaStreamSynchronize(s) == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in 1D init");
  }

  double time_of(long long n) const { return (double)n * g.dt; }
  double z_lo() const { return g.z0 + g.lo * g.dz; }
  double z_hi() const { return g.z0 + g.hi * g.dz; }
  long long rows_inside(double t) const { return (long long)std::ceil((z_hi() + beta * kC * t) / lat.h - 0.5); }

  int alloc_parts(long n) {
    for (int b = 0; b < 2; b++) {
      Parts1<T>& q = P2[b];
      q.z = dal<double>(n); q.ux = dal<T>(n); q.uy = dal<T>(n); q.uz = dal<T>(n); q.w = dal<T>(n);
      q.id = dal<uint32_t>(n);
      if (!q.z || !q.ux || !q.uy || !q.uz || !q.w || !q.id) return PIC_ENOMEM;
    }
    blk = dal<int>(n / 256 + 2);
    if (!blk) return PIC_ENOMEM;
    cap = n;
    return PIC_OK;
  }

  int grow(long need) {
    const long ncap = std::max(need + need / 2, 2 * cap);
    const Parts1<T> o = P2[cur];
    Parts1<T> keep = o;
    if (alloc_parts(ncap) != PIC_OK) return fail(PIC_ENOMEM, "particle allocation failed");
    if (count_ub > 0) {
      const Parts1<T>& d = P2[cur];
      cudaMemcpyAsync(d.z, keep.z, 8 * (size_t)count_ub, cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(d.ux, keep.ux, sizeof(T) * count_ub, cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(d.uy, keep.uy, sizeof(T) * count_ub, cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(d.uz, keep.uz, sizeof(T) * count_ub, cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(d.w, keep.w, sizeof(T) * count_ub, cudaMemcpyDeviceToDevice, s);
      cudaMemcpyAsync(d.id, keep.id, 4 * (size_t)count_ub, cudaMemcpyDeviceToDevice, s);
    }
    return PIC_OK;
  }

  int read_count() {
    Ctrl1 h{};
    cudaMemcpyAsync(&h, ctrl, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) return -1;
    return h.count;
  }

  int compact() {
    const int n_old = (int)count_ub;
    if (n_old <= 0) return PIC_OK;
    const int nb = (int)nb1(n_old, 256);
    k1_live_per_block<T><<<nb, 256, 0, s>>>(P2[cur], ctrl, blk);
    k1_scan_blocks<<<1, 1024, 0, s>>>(blk, nb, ctrl);
    k1_scatter<T><<<nb, 256, 0, s>>>(P2[cur], P2[1 - cur], blk, n_old);
    nl += 3;
    cur = 1 - cur;
    const int c = read_count();
    if (c < 0) return fail(PIC_ECUDA, "CUDA error in compaction");
    count_ub = c;
    compactions++;
    return PIC_OK;
  }

  // rows [m0, m1) enter at time t: their slots are taken now, their state is written by the next step's k1_push, or by
  // k1_inject (store_rows) before anything else reads or moves the particles
  int inject(long long m0, long long m1, double t) {
    if (m1 <= m0) return PIC_OK;
    const long nrow = (long)(m1 - m0);
    if (store_rows() != PIC_OK) return st;
    if (count_ub + nrow > cap && grow(count_ub + nrow) != PIC_OK) return st;
    pend.m0 = m0; pend.nrow = (int)nrow; pend.at = (int)count_ub; pend.t = t; pend.zlo = z_lo();
    count_ub += nrow;
    return PIC_OK;
  }

  int store_rows() {
    if (pend.nrow == 0) return PIC_OK;
    k1_inject<T><<<nb1(pend.nrow, 128), 128, 0, s>>>(P2[cur], ctrl, lat, pend);
    nl++;
    pend.nrow = 0;
    return cudaGetLastError() == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in 1D inflow");
  }

  int load_plasma(const pic_plasma* p) override {
    if (st != PIC_OK) return st;
    if (loaded) return fail(PIC_ESTATE, "plasma already loaded");
    if (p->ppc_z < 1 || p->n0 < 0) return fail(PIC_EINVAL, "bad plasma");
    if (p->beam_n > 0) return fail(PIC_EINVAL, "1D: no test beam");
    lat.h = g.dz / p->ppc_z;
    lat.gamma = gamma; lat.beta = beta;
    lat.n0 = p->n0; lat.z_start_lab = p->z_start_lab; lat.ramp_lab = p->ramp_lab; lat.length_lab = p->length_lab;
    lat.dz = g.dz; lat.ppc = p->ppc_z;
    ions = p->ions != 0;
    const double t = time_of(step);
    const long long m_end = rows_inside(t);
    const long long m_beg = (long long)std::ceil((z_lo() + beta * kC * t) / lat.h - 0.5);
    const long want = (long)(m_end - m_beg) * 2 + 4096;
    if (alloc_parts(want) != PIC_OK) return fail(PIC_ENOMEM, "particle allocation failed");
    count_ub = 0;
    if (inject(m_beg, m_end, t) != PIC_OK || store_rows() != PIC_OK) return st;
    row_next = m_end;
    mlo = m_beg;
    loaded = true;
    return cudaStreamSynchronize(s) == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in plasma load");
  }

  int set_laser(const pic_laser* l) override {
    if (st != PIC_OK) return st;
    if (!(l->lambda0 > 0) || !(l->tau_fwhm > 0)) return fail(PIC_EINVAL, "bad laser");
    if (l->beta_s != 0.0) return fail(PIC_EINVAL, "1D antenna: the plane is at rest in the computational frame");
    las = *l;
    has_laser = true;
    return PIC_OK;
  }

  // the lab waveform E0 exp(-(s - t_peak)^2/(2 sigma^2)) sin(omega (s - t_peak) + phase) emitted from a plane
  // at rest: amplitude and time scaled by (1 + beta) gamma (Sec. 3.1.2, PR-14)
  double emit(double tp) const {
    const double om = 2.0 * kPi * kC / las.lambda0;
    const double E0 = las.a0 * kMe * kC * om / kQe;
    const double dop = (1.0 + beta) * gamma;
    const double sl = tp / dop;
    const double sig = las.tau_fwhm / (2.0 * std::sqrt(std::log(2.0)));
    const double u = sl - las.t_peak;
    return E0 * std::exp(-u * u / (2.0 * sig * sig)) * std::sin(om * u + las.phase) / dop;
  }

  static double shape_h(int order, double s) {
    const double a = std::fabs(s);
    if (order == 1) return a < 1.0 ? 1.0 - a : 0.0;
    if (a < 1.0) return 2.0 / 3.0 - a * a + 0.5 * a * a * a;
    if (a < 2.0) { const double t = 2.0 - a; return t * t * t / 6.0; }
    return 0.0;
  }

  // event pairs around the timed launches, read when the timing is queried (no wait inside the step)
  void tbeg(int which) {
    if (!(timing_on && timing_which == which)) return;
    cudaEvent_t a, b;
    cudaEventCreate(&a);
    cudaEventCreate(&b);
    cudaEventRecord(a, s);
    tev.push_back(a);
    tev.push_back(b);
  }
  void tend(int which) {
    if (!(timing_on && timing_which == which) || tev.empty()) return;
    cudaEventRecord(tev.back(), s);
    t_n++;
  }
  void tcollect() {
    if (tev.empty()) return;
    cudaEventSynchronize(tev.back());
    for (size_t i = 0; i + 1 < tev.size(); i += 2) {
      float ms = 0;
      cudaEventElapsedTime(&ms, tev[i], tev[i + 1]);
      t_ms += ms;
    }
    for (auto e : tev) cudaEventDestroy(e);
    tev.clear();
  }

  // a kernel that may begin launching while the one before it on the stream ends (it waits for it on the device)
  template <class... KA, class... A>
  void chain(void (*k)(KA...), unsigned blocks, unsigned threads, const A&... args) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(blocks);
    c.blockDim = dim3(threads);
    c.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    c.attrs = at;
    c.numAttrs = 1;
    cudaLaunchKernelEx(&c, k, KA(args)...);
    nl++;
  }

  // moving window (lab frame): the grid moves down by whole cells at the start of a step
  int window_shift() {
    if (!cfg.moving_window) return 0;
    const long long want = (long long)std::floor(cfg.window_beta * kC * time_of(step) / g.dz);
    const long long sh = want - shifts;
    if (sh <= 0) return 0;
    shifts = want;
    g.z0 = want * g.dz;
    return (int)std::min<long long>(sh, g.nz + 1);
  }

  // the fields between two pushes: Ampère of the step before (ampere), the window's shift, Faraday, the Friedman
  // history and the gather copies of the step to come (faraday)
  void fields(bool ampere, bool faraday, int shift) {
    const double th = cfg.theta;
    Fields1<T> a;
    a.in = fs2[fc]; a.out = fs2[1 - fc];
    a.J = J2[jc]; a.Jz = J2[1 - jc];
    a.fE = fE; a.fB = fB;
    a.c1 = T(1.0 + th / 4.0); a.c2 = T(0.5); a.c3 = T(0.5 - th / 4.0);
    a.ha = T(1.0 - th / 2.0); a.hb = T(th / 2.0);
    a.dt = T(g.dt); a.idz = T(g.idz); a.c2idz = T(kC * kC * g.idz); a.ie0 = T(1.0 / kEps0);
    a.ampere = ampere; a.faraday = faraday;
    a.filt_j = cfg.filter_J && P > 0; a.filt_g = cfg.filter_gather && P > 0; a.nodal = nodal;
    a.shift = shift;
    a.H = a.filt_j || a.filt_g ? taps.P * taps.s : 0;
    tbeg(1);
    chain(k1_fields<T>, nb1(g.nz + 1, NT1), FB1, g, pm, taps, a);
    tend(1);
    fc = 1 - fc;
    if (faraday) jc = 1 - jc;   // the next deposit goes to the current just set to zero
  }

  template <int ORD, bool MC>
  void launch_push(const Ions1& io, const Ant1& an) {
    constexpr int PB1 = push_threads1<T>();
    const unsigned nbp = std::max(1u, nb1(count_ub, PB1));
    const unsigned nbi = io.on ? nb1(g.nz + 1, PB1 / 32) : 0;
    chain(k1_push<T, ORD, MC>, nbp + nbi, PB1, g, fE, fB, J2[jc], P2[cur], (int)count_ub, ctrl,
          T(-kQe * g.dt / (2.0 * kMe)), T(-kQe), z_lo(), z_hi() + g.dz, lat, pend, io, an, (int)nbp);
    pend.nrow = 0;
  }

  // push of the electrons (with the rows that entered at the end of the last step), ions, antenna, inflow
  int particles() {
    const double tn = time_of(step), tn1 = time_of(step + 1);
    // ions fixed in the lab: no current in the lab frame (beta = 0)
    Ions1 io{};
    io.on = loaded && ions && row_next > mlo && beta > 0.0;
    io.mlo = mlo; io.mhi = row_next; io.t0 = tn; io.t1 = tn1;
    Ant1 a{};
    if (has_laser && las.z_antenna >= z_lo() && las.z_antenna < z_hi()) {
      const double Z = (las.z_antenna - g.z0) / g.dz;
      const int f = (int)std::floor(Z);
      const double K = -2.0 * kEps0 * kC * emit(0.5 * (tn + tn1));
      a.on = 1;
      a.k0 = f - 3;
      for (int i = 0; i < 8; i++) a.v[i] = K * shape_h(cfg.shape_order, Z - (a.k0 + i)) / g.dz;
    }
    tbeg(0);
    if (cfg.shape_order == 3) {
      if (nodal) launch_push<3, true>(io, a);
      else launch_push<3, false>(io, a);
    } else {
      if (nodal) launch_push<1, true>(io, a);
      else launch_push<1, false>(io, a);
    }
    tend(0);
    step++;
    // ion rows that left, plasma rows entering through z_hi
    if (loaded) {
      while (mlo < row_next && (mlo + 0.5) * lat.h - beta * kC * tn1 < z_lo()) mlo++;
      const long long m_end = rows_inside(tn1);
      if (m_end > row_next) {
        if (inject(row_next, m_end, tn1) != PIC_OK) return st;
        row_next = m_end;
      }
      // the dead slots (left the domain, or rows without plasma) are squeezed out now and then
      if (count_ub > 65536 && (step & 63) == 0) {
        if (store_rows() != PIC_OK || compact() != PIC_OK) return st;
      }
    }
    return PIC_OK;
  }

  int run(int nsteps) override {
    if (st != PIC_OK) return st;
    int r = PIC_OK;
    for (int q = 0; q < nsteps && r == PIC_OK; q++) {
      fields(q > 0, true, window_shift());
      r = particles();
    }
    // the last step's Ampère and inflow, so that the state is whole between calls
    if (nsteps > 0) fields(true, false, 0);
    if (store_rows() != PIC_OK || r != PIC_OK) return st;
    return cudaGetLastError() == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in 1D step");
  }

  int sync() override {
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(PIC_ECUDA, "CUDA error");
    return st;
  }

  int btd_set(const pic_btd_req*) override { return fail(PIC_EINVAL, "1D: no boosted-to-lab samples"); }
  int btd_get(pic_btd_out*) override { return fail(PIC_EINVAL, "1D: no boosted-to-lab samples"); }

  T* comp_ptr(int comp) {
    const int n = g.n1p;
    if (comp < 3) return fs2[fc].E + comp * n;
    if (comp < 6) return fs2[fc].B + (comp - 3) * n;
    return J2[jc] + (comp - 6) * n;
  }

  int get_field(int comp, double* dst, int on_device) override {
    if (comp < 0 || comp > PIC_RHO) return fail(PIC_EINVAL, "bad component");
    const int n1 = g.nz + 1;
    if (on_device && !ddst.order(s)) return fail(PIC_ECUDA, "CUDA error in get_field");
    if (comp == PIC_RHO) {
      cudaMemsetAsync(rho, 0, sizeof(double) * g.n1p, s);
      if (loaded && count_ub > 0) {
        k1_rho_e<T><<<nb1(count_ub, 128), 128, 0, s>>>(g, P2[cur], ctrl, cfg.shape_order, rho);
        nl++;
      }
      if (loaded && ions && row_next > mlo) {
        k1_rho_i<<<nb1(n1, 128), 128, 0, s>>>(g, lat, cfg.shape_order, mlo, row_next, time_of(step), rho);
        nl++;
      }
      cudaMemcpyAsync(dst, rho, sizeof(double) * n1, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s);
    } else {
      // written in place where a kernel may, else through the scratch
      double* out = on_device && DeviceDst::in_place(dst) ? dst : outd;
      k1_out<T><<<nb1(n1, 256), 256, 0, s>>>(n1, comp_ptr(comp), out);
      nl++;
      if (out != dst)
        cudaMemcpyAsync(dst, outd, sizeof(double) * n1, on_device ? cudaMemcpyDeviceToDevice : cudaMemcpyDeviceToHost, s);
    }
    return cudaStreamSynchronize(s) == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in get_field");
  }

  int set_field(int comp, const double* src) override {
    if (comp < 0 || comp > 8) return fail(PIC_EINVAL, "bad component");
    const int n1 = g.nz + 1;
    cudaMemcpyAsync(outd, src, sizeof(double) * n1, cudaMemcpyHostToDevice, s);
    k1_in<T><<<nb1(n1, 256), 256, 0, s>>>(n1, outd, comp_ptr(comp));
    nl++;
    return cudaStreamSynchronize(s) == cudaSuccess ? PIC_OK : fail(PIC_ECUDA, "CUDA error in set_field");
  }

  int get_particles(int species, double* x, double* y, double* z, double* ux, double* uy, double* uz, double* w,
                    uint32_t* id, int32_t* flags, int64_t* count) override {
    if (species != 0) return fail(PIC_EINVAL, "1D: electrons only (the ions are a column current)");
    if (!loaded) { if (count) *count = 0; return PIC_OK; }
    // live electrons in slot order
    const int c = read_count();
    if (c < 0) return fail(PIC_ECUDA, "CUDA error");
    std::vector<double> hz(c);
    std::vector<T> hux(c), huy(c), huz(c), hw(c);
    std::vector<uint32_t> hid(c);
    const Parts1<T>& p = P2[cur];
    if (c > 0) {
      cudaMemcpyAsync(hz.data(), p.z, 8 * (size_t)c, cudaMemcpyDeviceToHost, s);
      cudaMemcpyAsync(hux.data(), p.ux, sizeof(T) * c, cudaMemcpyDeviceToHost, s);
      cudaMemcpyAsync(huy.data(), p.uy, sizeof(T) * c, cudaMemcpyDeviceToHost, s);
      cudaMemcpyAsync(huz.data(), p.uz, sizeof(T) * c, cudaMemcpyDeviceToHost, s);
      cudaMemcpyAsync(hw.data(), p.w, sizeof(T) * c, cudaMemcpyDeviceToHost, s);
      cudaMemcpyAsync(hid.data(), p.id, 4 * (size_t)c, cudaMemcpyDeviceToHost, s);
      if (cudaStreamSynchronize(s) != cudaSuccess) return fail(PIC_ECUDA, "CUDA error");
    }
    int64_t o = 0;
    const bool want = x || y || z || ux || uy || uz || w || id || flags;
    for (int j = 0; j < c; j++) {
      if (!(hw[j] > T(0))) continue;
      if (want) {
        if (x) x[o] = 0.0;
        if (y) y[o] = 0.0;
        if (z) z[o] = hz[j];
        if (ux) ux[o] = (double)hux[j];
        if (uy) uy[o] = (double)huy[j];
        if (uz) uz[o] = (double)huz[j];
        if (w) w[o] = (double)hw[j];
        if (id) id[o] = hid[j];
        if (flags) flags[o] = 1;
      }
      o++;
    }
    if (count) *count = o;
    return PIC_OK;
  }

  int stats(pic_stats* o) override {
    double trap = o->trap_gamma_lab > 0.0 ? o->trap_gamma_lab : 0.0;
    if (trap == 0.0 && has_laser && loaded && lat.n0 > 0.0) {
      const double wp = std::sqrt(lat.n0 * kQe * kQe / (kEps0 * kMe));
      trap = 2.0 * (2.0 * kPi * kC / las.lambda0) / wp;
    }
    cudaMemsetAsync(sred, 0, 4 * sizeof(double), s);
    Parts1<T> p = P2[cur];
    if (!loaded) cudaMemsetAsync(ctrl, 0, sizeof(Ctrl1), s);
    k1_stats<T><<<64, 256, 0, s>>>(g, fs2[fc].E, fs2[fc].B, p, ctrl, gamma, beta, trap, sred);
    nl++;
    double h[4];
    cudaMemcpyAsync(h, sred, sizeof(h), cudaMemcpyDeviceToHost, s);
    if (cudaStreamSynchronize(s) != cudaSuccess) return fail(PIC_ECUDA, "CUDA error in stats");
    o->step = step; o->t = time_of(step);
    o->dt = g.dt; o->dx = 0.0; o->dz = g.dz; o->gamma = gamma; o->beta = beta;
    o->n_electrons = loaded ? (int64_t)h[0] : 0;
    o->n_beam_active = 0; o->beam_gamma_lab = 0.0; o->beam_spread = 0.0;
    o->field_energy = h[1];
    o->gx_lo = 0; o->gx_hi = 0; o->gz_lo = g.lo; o->gz_hi = g.hi;
    o->sorts = compactions; o->overflow_chunks = 0;
    o->z0 = g.z0;
    o->trap_gamma_lab = trap;
    o->trapped_charge = kQe * h[2];
    return PIC_OK;
  }

  int64_t launches() const override { return nl; }

  int kernel_timing(int enable, int which, double* ms_total, int64_t* n) override {
    if (which != 0 && which != 1) return PIC_EINVAL;
    if (!ev0) { cudaEventCreate(&ev0); cudaEventCreate(&ev1); }
    tcollect();
    if (enable >= 0) {
      timing_on = enable != 0;
      timing_which = which;
      if (enable) { t_ms = 0; t_n = 0; }
    }
    if (ms_total) *ms_total = t_ms;
    if (n) *n = t_n;
    return PIC_OK;
  }

  int status() const override { return st; }
  const std::string& error() const override { return err; }

 private:
  pic_config cfg;
  pic_alloc_fn alloc;
  pic_free_fn freef;
  void* user;
  cudaStream_t s;
  std::vector<std::pair<void*, size_t>> allocs;
  int st = PIC_OK;
  std::string err;
  G1 g{};
  double gamma = 1.0, beta = 0.0;
  int P = 0;
  bool nodal = false;
  Taps1<T> taps{};
  Pml1<T> pm{};
  Set1<T> fs2[2]{};      // the current fields are fs2[fc], the step's current J2[jc]
  T* J2[2] = {nullptr, nullptr};
  int fc = 0, jc = 0;
  T *fE = nullptr, *fB = nullptr;
  double *rho = nullptr, *outd = nullptr, *sred = nullptr;
  Ctrl1* ctrl = nullptr;
  Parts1<T> P2[2]{};
  int cur = 0;
  int* blk = nullptr;
  long cap = 0;
  long count_ub = 0;
  Rows1 pend{};          // rows whose slots are taken and whose state is not yet stored
  bool loaded = false, ions = false, has_laser = false;
  Lat1 lat{};
  pic_laser las{};
  long long row_next = 0, mlo = 0, shifts = 0, step = 0;
  int64_t nl = 0, compactions = 0;
  DeviceDst ddst;        // get_field to device memory
  bool timing_on = false;
  int timing_which = 0;
  double t_ms = 0;
  std::vector<cudaEvent_t> tev;
  int64_t t_n = 0;
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
};

}  // namespace

Sim3Api* make_sim1(const pic_config* cfg, pic_alloc_fn alloc, pic_free_fn free_fn, void* user, cudaStream_t s,
                   int* status, std::string* err) {
  Sim3Api* r = nullptr;
  int st = PIC_OK;
  if (cfg->precision == PIC_FP64) {
    auto* p = new Sim1<double>(*cfg, alloc, free_fn, user, s);
    st = p->init();
    if (st != PIC_OK) { if (err) *err = p->error(); delete p; } else r = p;
  } else {
    auto* p = new Sim1<float>(*cfg, alloc, free_fn, user, s);
    st = p->init();
    if (st != PIC_OK) { if (err) *err = p->error(); delete p; } else r = p;
  }
  if (status) *status = st;
  return r;
}

}  // namespace picgb
