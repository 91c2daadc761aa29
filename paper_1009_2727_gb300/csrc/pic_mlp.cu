// Multilayer perceptron for the stage surrogate: widths w0 -> w1 -> ... -> wL,
// GELU between layers and a linear output. Weights are kept as FP32 master
// copies (AdamW) and BF16 compute copies; activations are stored in BF16; every
// product accumulates in FP32. One tiled GEMM kernel serves the forward pass
// (X W^T), the weight gradient (dZ^T H) and the input gradient (dZ W).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <vector>

#include "../../include/pic.h"

namespace {

constexpr int GT = 64;    // output tile (rows and columns)
constexpr int GK = 16;    // reduction slice

__device__ __forceinline__ float ld_el(const float* p, long i) { return p[i]; }
__device__ __forceinline__ float ld_el(const __nv_bfloat16* p, long i) { return __bfloat162float(p[i]); }

// C(m, n) = sum_k A(m, k) B(k, n) (+ bias[n]); A(m, k) = TA ? A[k lda + m] : A[m lda + k],
// B(k, n) = TB ? B[n ldb + k] : B[k ldb + n]. 256 threads, 64 x 64 tile, 4 x 4 outputs per thread.
// EPI 0: store C (FP32); EPI 1: store Z = C + bias (FP32) and H = GELU(Z) (BF16); EPI 2: store C + bias.
template <class TAe, class TBe, bool TA, bool TB, int EPI>
__global__ void __launch_bounds__(256) k_gemm(int M, int N, int K, const TAe* A, int lda, const TBe* B, int ldb,
                                              float* C, int ldc, const float* bias, __nv_bfloat16* H) {
  __shared__ float As[GK][GT + 1];
  __shared__ float Bs[GK][GT + 1];
  const int tx = threadIdx.x & 15, ty = threadIdx.x >> 4;
  const int m0 = blockIdx.y * GT, n0 = blockIdx.x * GT;
  float acc[4][4] = {};
  for (int k0 = 0; k0 < K; k0 += GK) {
    for (int e = threadIdx.x; e < GK * GT; e += 256) {
      const int kk = e / GT, mm = e - kk * GT;
      const int m = m0 + mm, n = n0 + mm, k = k0 + kk;
      float a = 0.0f, b = 0.0f;
      if (m < M && k < K) a = TA ? ld_el(A, (long)k * lda + m) : ld_el(A, (long)m * lda + k);
      if (n < N && k < K) b = TB ? ld_el(B, (long)n * ldb + k) : ld_el(B, (long)k * ldb + n);
      As[kk][mm] = a;
      Bs[kk][mm] = b;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < GK; kk++) {
      float av[4], bv[4];
#pragma unroll
      for (int i = 0; i < 4; i++) { av[i] = As[kk][ty + 16 * i]; bv[i] = Bs[kk][tx + 16 * i]; }
#pragma unroll
      for (int i = 0; i < 4; i++)
#pragma unroll
        for (int j = 0; j < 4; j++) acc[i][j] += av[i] * bv[j];
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; i++)
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m >= M || n >= N) continue;
      float v = acc[i][j];
      if (EPI >= 1) v += bias[n];
      C[(long)m * ldc + n] = v;
      if (EPI == 1) H[(long)m * ldc + n] = __float2bfloat16(0.5f * v * (1.0f + erff(v * 0.70710678118654752f)));
    }
}

// dZ = dH * GELU'(Z), GELU'(z) = Phi(z) + z phi(z)
__global__ void k_gelu_back(long n, const float* Z, const float* dH, float* dZ) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float z = Z[i];
  const float d = 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
  dZ[i] = dH[i] * d;
}

// db[j] = sum_i dZ[i, j] (one block per column)
__global__ void k_colsum(int n, int cols, const float* dZ, float* db) {
  __shared__ float red[256];
  const int j = blockIdx.x;
  float s = 0.0f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += dZ[(long)i * cols + j];
  red[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) db[j] = red[0];
}

// mean squared error over n x d outputs; dY = 2 (Y - T) / (n d); loss summed into *loss
// loss: the sum is added to loss[*eidx] when eidx is given (the epoch's slot of a training run), else to *loss
__global__ void k_mse(long nd, const float* Y, const float* T, float* dY, float* loss, const int* eidx) {
  __shared__ float red[256];
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  float l = 0.0f;
  if (i < nd) {
    const float e = Y[i] - T[i];
    dY[i] = 2.0f * e / (float)nd;
    l = e * e / (float)nd;
  }
  red[threadIdx.x] = l;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) atomicAdd(eidx ? loss + *eidx : loss, red[0]);
}

__global__ void k_to_bf16(long n, const float* src, __nv_bfloat16* dst) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = __float2bfloat16(src[i]);
}

// AdamW (decoupled weight decay) on the FP32 master parameters, then their BF16 copies. The bias corrections
// c1 = 1 - b1^t, c2 = 1 - b2^t come as arguments, or (ctab given) from a host-computed table at step
// (*eidx) * nbat + kk: the form a captured epoch replays
__global__ void k_adamw(long n, float* p, const float* g, float* m, float* v, __nv_bfloat16* pb, float lr, float b1,
                        float b2, float eps, float wd, float c1, float c2, const float2* ctab, const int* eidx,
                        int nbat, int kk) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (ctab) {
    const float2 c = ctab[(long)(*eidx) * nbat + kk];
    c1 = c.x;
    c2 = c.y;
  }
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  const float pi = p[i] - lr * ((mi / c1) / (sqrtf(vi / c2) + eps) + wd * p[i]);
  p[i] = pi;
  pb[i] = __float2bfloat16(pi);
}

// rows idx[i] of X (n x dx) and T (n x dt) into contiguous batches
__global__ void k_gather_rows(int nb, const int* idx, const float* X, int dx, const float* T, int dt, float* Xb,
                              float* Tb) {
  const int r = blockIdx.x;
  if (r >= nb) return;
  const long s = idx[r];
  for (int j = threadIdx.x; j < dx; j += blockDim.x) Xb[(long)r * dx + j] = X[s * dx + j];
  for (int j = threadIdx.x; j < dt; j += blockDim.x) Tb[(long)r * dt + j] = T[s * dt + j];
}

// ---------------------------------------------------------------------------
// Small batches (training minibatches, up to SB_ROWS rows). At 64 rows and widths of 256 a minibatch is 0.05 us of FP32
// work on the whole GPU, so what counts is how many SMs share a product and how many dependent launches there are:
// 64 x 64 tiles gave each product 4 CTAs and 14-34 us, and 21 launches made 240 us of a minibatch. Here a product is
// cut into 8 x 16 output tiles (128 CTAs for 64 x 256), one output per thread, its sum taken in the order of the large
// tiles (the results are bitwise theirs); the row gather, BF16 rounding, bias, GELU, loss and GELU' ride with the
// products, and one launch takes the gradients and AdamW of every layer: 8 launches for four layers. Consecutive
// launches overlap their start (programmatic dependent launch): each kernel fetches what its predecessor does not write
// (weights, pre-activations, moments) before it waits for it.
// Measured (6-256-256-256-4, batch 64): 235 -> 33 us a minibatch; each product 5.4-6.8 us alone, the gradients 9.3 us
// (19.5 us with element-wise staging and the bias sums from global memory): bound by the eight launches' latencies.
constexpr int SB_ROWS = 512;    // above: the 64 x 64 tiles, which re-read less
constexpr int SB_M = 8;         // output tile: rows
constexpr int SB_N = 16;        //              columns
constexpr int SB_KC = 256;      // reduction slice held in shared memory (FP32)
constexpr int SB_LD = SB_KC + 4;   // rows 16 bytes apart modulo 128: the 16-byte reads of eight rows hit all banks
constexpr int SB_THREADS = SB_M * SB_N;

// eight BF16 values of a row from p[k ..] (zero past K), read through L2 (what a kernel fetches before its wait must not
// come from an older L1 line); vec: 16-byte loads are aligned and K is a multiple of 8
__device__ __forceinline__ uint4 ld8(const __nv_bfloat16* p, int k, int K, bool vec) {
  if (vec && k + 8 <= K) return __ldcg(reinterpret_cast<const uint4*>(p + k));
  __align__(16) __nv_bfloat16 v[8];
#pragma unroll
  for (int q = 0; q < 8; q++) v[q] = k + q < K ? __ldcg(p + k + q) : __float2bfloat16(0.0f);
  return *reinterpret_cast<const uint4*>(v);
}
__device__ __forceinline__ void unpack8(const uint4& u, float* f) {
  const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
  for (int q = 0; q < 4; q++) {
    f[2 * q] = __uint_as_float(w[q] << 16);
    f[2 * q + 1] = __uint_as_float(w[q] & 0xffff0000u);
  }
}
__device__ __forceinline__ void put8(float* d, const float* f) {
  reinterpret_cast<float4*>(d)[0] = make_float4(f[0], f[1], f[2], f[3]);
  reinterpret_cast<float4*>(d)[1] = make_float4(f[4], f[5], f[6], f[7]);
}

// acc += sum over the staged slice of a row times a row, in order
__device__ __forceinline__ void slice_dot(const float* a, const float* b, int kn, float& acc) {
#pragma unroll 8
  for (int k = 0; k < kn; k += 4) {
    const float4 x = *reinterpret_cast<const float4*>(a + k), y = *reinterpret_cast<const float4*>(b + k);
    acc += x.x * y.x;
    acc += x.y * y.y;
    acc += x.z * y.z;
    acc += x.w * y.w;
  }
}

// one layer's forward product of M rows: Z = H W^T + b. FIRST: H is the BF16 rounding of the rows idx[r] (or r) of the
// FP32 inputs x. Hidden layers store Z (FP32) and GELU(Z) (BF16); the last layer (LAST) stores Z and, with targets t,
// the gradient dY = 2 (Z - t[idx[r]]) / (M N) of the mean squared error and every output's share of it (sq).
template <bool FIRST, bool LAST>
__global__ void __launch_bounds__(SB_THREADS) k_sb_fwd(int M, int N, int K, const __nv_bfloat16* H, const float* x,
                                                       const int* idx, const __nv_bfloat16* W, const float* bias,
                                                       float* Z, __nv_bfloat16* Hn, const float* t, float* dY,
                                                       float* sq, int vec) {
  __shared__ __align__(16) float sa[SB_M][SB_LD], sw[SB_N][SB_LD];
  const int tid = threadIdx.x, ty = tid / SB_N, tx = tid % SB_N;
  const int m0 = blockIdx.y * SB_M, n0 = blockIdx.x * SB_N;
  auto stage_w = [&](int k0) {
    for (int e = tid; e < SB_N * (SB_KC / 8); e += SB_THREADS) {
      const int r = e / (SB_KC / 8), k = k0 + (e % (SB_KC / 8)) * 8;
      uint4 u = make_uint4(0, 0, 0, 0);
      if (n0 + r < N && k < K) u = ld8(W + (long)(n0 + r) * K, k, K, vec);
      float f[8];
      unpack8(u, f);
      put8(&sw[r][k - k0], f);
    }
  };
  // the weights were last written before the predecessor began (the first layer's predecessor is their update)
  if (!FIRST) stage_w(0);
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  float acc = 0.0f;
  for (int k0 = 0; k0 < K; k0 += SB_KC) {
    if (FIRST || k0 > 0) stage_w(k0);
    for (int e = tid; e < SB_M * (SB_KC / 8); e += SB_THREADS) {
      const int r = e / (SB_KC / 8), k = k0 + (e % (SB_KC / 8)) * 8, m = m0 + r;
      float f[8] = {};
      if (m < M && k < K) {
        if (FIRST) {
          const float* xr = x + (long)(idx ? idx[m] : m) * K;
#pragma unroll
          for (int q = 0; q < 8; q++) f[q] = k + q < K ? __bfloat162float(__float2bfloat16(xr[k + q])) : 0.0f;
        } else {
          unpack8(ld8(H + (long)m * K, k, K, vec), f);
        }
      }
      put8(&sa[r][k - k0], f);
    }
    __syncthreads();
    slice_dot(sa[ty], sw[tx], min(SB_KC, (K - k0 + 3) & ~3), acc);
    __syncthreads();
  }
  const int m = m0 + ty, n = n0 + tx;
  if (m >= M || n >= N) return;
  const long o = (long)m * N + n;
  const float z = acc + bias[n];
  Z[o] = z;
  if (!LAST) Hn[o] = __float2bfloat16(0.5f * z * (1.0f + erff(z * 0.70710678118654752f)));
  if (LAST && t) {
    const float nd = (float)((long)M * N), d = z - t[(long)(idx ? idx[m] : m) * N + n];
    dY[o] = 2.0f * d / nd;
    sq[o] = d * d / nd;
  }
}

// input gradient through the GELU of the layer below: dZ'(m, i) = (sum_o dZ(m, o) W(o, i)) GELU'(Z'(m, i)),
// GELU'(z) = Phi(z) + z phi(z); M rows, K outputs o, N inputs i
__global__ void __launch_bounds__(SB_THREADS) k_sb_dx(int M, int N, int K, const float* dZ, const __nv_bfloat16* W,
                                                      const float* Zl, float* dZl, int vec, int vecz) {
  __shared__ __align__(16) float sa[SB_M][SB_LD], sw[SB_N][SB_LD];   // sw: the weights' columns as rows
  const int tid = threadIdx.x, ty = tid / SB_N, tx = tid % SB_N;
  const int m0 = blockIdx.y * SB_M, n0 = blockIdx.x * SB_N;
  auto stage_w = [&](int k0) {
    for (int e = tid; e < SB_KC * (SB_N / 8); e += SB_THREADS) {
      const int k = e % SB_KC, c = (e / SB_KC) * 8;
      uint4 u = make_uint4(0, 0, 0, 0);
      if (k0 + k < K && n0 + c < N) u = ld8(W + (long)(k0 + k) * N, n0 + c, N, vec);
      float f[8];
      unpack8(u, f);
#pragma unroll
      for (int q = 0; q < 8; q++) sw[c + q][k] = f[q];
    }
  };
  // weights and pre-activations were written before the predecessor began
  stage_w(0);
  const int m = m0 + ty, n = n0 + tx;
  const float z = m < M && n < N ? __ldcg(Zl + (long)m * N + n) : 0.0f;
  const float d = 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  float acc = 0.0f;
  for (int k0 = 0; k0 < K; k0 += SB_KC) {
    if (k0 > 0) stage_w(k0);
    for (int e = tid; e < SB_M * (SB_KC / 4); e += SB_THREADS) {
      const int r = e / (SB_KC / 4), k = k0 + (e % (SB_KC / 4)) * 4, mr = m0 + r;
      float4 f = make_float4(0.f, 0.f, 0.f, 0.f);
      if (mr < M && k < K) {
        const float* p = dZ + (long)mr * K + k;
        if (vecz && k + 4 <= K) {
          f = *reinterpret_cast<const float4*>(p);
        } else {
          f.x = p[0];
          if (k + 1 < K) f.y = p[1];
          if (k + 2 < K) f.z = p[2];
          if (k + 3 < K) f.w = p[3];
        }
      }
      *reinterpret_cast<float4*>(&sa[r][k - k0]) = f;
    }
    __syncthreads();
    slice_dot(sa[ty], sw[tx], min(SB_KC, (K - k0 + 3) & ~3), acc);
    __syncthreads();
  }
  if (m < M && n < N) dZl[(long)m * N + n] = acc * d;
}

// AdamW's constants; the bias corrections c1 = 1 - b1^t, c2 = 1 - b2^t come from a host-computed table at step
// (*eidx) * nbat + kk (the form a captured epoch replays)
struct AdamC {
  float lr, b1, b2, eps, wd;
  const float2* ctab;
  const int* eidx;
  int nbat, kk;
};

__device__ __forceinline__ float adamw_one(float pi, float gi, float& m, float& v, const AdamC& a, float2 c) {
  // roundings written out, so that this is k_adamw bit for bit
  m = fmaf(1.0f - a.b1, gi, __fmul_rn(a.b1, m));
  v = fmaf(__fmul_rn(1.0f - a.b2, gi), gi, __fmul_rn(a.b2, v));
  return fmaf(-a.lr, fmaf(a.wd, pi, (m / c.x) / (sqrtf(v / c.y) + a.eps)), pi);
}

struct SbLayer {
  const float* dZ;            // M x N
  const __nv_bfloat16* H;     // M x K (layers above the first)
  long off_w, off_b;
  int N, K, blocks, tk;       // tiles (tk along the inputs) end at block `blocks` of the launch
  int vz, vh;                 // four values of a row of dZ, of H load together (widths and bases aligned)
};
struct SbNet {
  SbLayer l[16];
  int L;
};

// gradients of every layer, dW(o, i) = sum_r dZ(r, o) H(r, i) and db(o) = sum_r dZ(r, o), on 32 x 32 tiles of the
// weights (rows summed in order); then AdamW and the BF16 copies (p given), or the gradient stored (g given). The first
// layer's H are the BF16-rounded rows idx[r] (or r) of x. The last
// block (a tile of the small last layer) sums the minibatch's loss, 256 outputs at a time.
constexpr int SB_GT = 32, SB_GR = 64;
__global__ void __launch_bounds__(256) k_sb_grad(SbNet net, int M, const float* x, const int* idx, float* p,
                                                 __nv_bfloat16* pb, float* mo, float* vo, float* g, AdamC a,
                                                 const float* sq, long nsq, float* loss) {
  __shared__ float sz[SB_GR][SB_GT + 1], sh[SB_GR][SB_GT + 1];   // padded: the bias sums read sz by columns
  __shared__ float red[256], sdb[SB_GT];
  int li = 0;
  while (li + 1 < net.L && (int)blockIdx.x >= net.l[li].blocks) li++;
  const SbLayer& L = net.l[li];
  const int b = (int)blockIdx.x - (li > 0 ? net.l[li - 1].blocks : 0);
  const int o0 = (b / L.tk) * SB_GT, i0 = (b % L.tk) * SB_GT;
  const int tid = threadIdx.x, ty = tid >> 4, tx = tid & 15;
  // the tile's parameters and moments were last written before the predecessors began
  float pv[2][2], mv[2][2], vv[2][2], bp = 0.f, bm = 0.f, bv = 0.f;
  const bool bias = i0 == 0 && tid < SB_GT && o0 + tid < L.N;
  float2 c = make_float2(1.0f, 1.0f);
  if (p) {
    c = __ldcg(a.ctab + (long)__ldcg(a.eidx) * a.nbat + a.kk);
#pragma unroll
    for (int u = 0; u < 2; u++)
#pragma unroll
      for (int w = 0; w < 2; w++) {
        const int o = o0 + ty + 16 * u, i = i0 + tx + 16 * w;
        pv[u][w] = mv[u][w] = vv[u][w] = 0.0f;
        if (o < L.N && i < L.K) {
          const long q = L.off_w + (long)o * L.K + i;
          pv[u][w] = __ldcg(p + q); mv[u][w] = __ldcg(mo + q); vv[u][w] = __ldcg(vo + q);
        }
      }
    if (bias) {
      const long q = L.off_b + o0 + tid;
      bp = __ldcg(p + q); bm = __ldcg(mo + q); bv = __ldcg(vo + q);
    }
  }
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
  float acc[2][2] = {};
  for (int r0 = 0; r0 < M; r0 += SB_GR) {
    const int nr = min(SB_GR, M - r0);
    // four values of a row of either operand per thread and pass, every load of the slice issued together
    constexpr int NP = SB_GR * SB_GT / 4 / 256;
    const int q = (tid & 7) * 4;
    float fz[NP][4], fh[NP][4];
#pragma unroll
    for (int u = 0; u < NP; u++) {
      const int r = (tid >> 3) + 32 * u, m = r0 + r;
#pragma unroll
      for (int j = 0; j < 4; j++) fz[u][j] = fh[u][j] = 0.0f;
      if (r >= nr) continue;
      const float* pz = L.dZ + (long)m * L.N + o0 + q;
      if (L.vz && o0 + q + 4 <= L.N) {
        const float4 f = *reinterpret_cast<const float4*>(pz);
        fz[u][0] = f.x; fz[u][1] = f.y; fz[u][2] = f.z; fz[u][3] = f.w;
      } else {
#pragma unroll
        for (int j = 0; j < 4; j++) if (o0 + q + j < L.N) fz[u][j] = pz[j];
      }
      if (li == 0) {
        const float* px = x + (long)(idx ? idx[m] : m) * L.K + i0 + q;
#pragma unroll
        for (int j = 0; j < 4; j++) if (i0 + q + j < L.K) fh[u][j] = __bfloat162float(__float2bfloat16(px[j]));
      } else {
        const __nv_bfloat16* ph = L.H + (long)m * L.K + i0 + q;
        if (L.vh && i0 + q + 4 <= L.K) {
          const uint2 w = *reinterpret_cast<const uint2*>(ph);
          fh[u][0] = __uint_as_float(w.x << 16); fh[u][1] = __uint_as_float(w.x & 0xffff0000u);
          fh[u][2] = __uint_as_float(w.y << 16); fh[u][3] = __uint_as_float(w.y & 0xffff0000u);
        } else {
#pragma unroll
          for (int j = 0; j < 4; j++) if (i0 + q + j < L.K) fh[u][j] = __bfloat162float(ph[j]);
        }
      }
    }
#pragma unroll
    for (int u = 0; u < NP; u++) {
      const int r = (tid >> 3) + 32 * u;
#pragma unroll
      for (int j = 0; j < 4; j++) { sz[r][q + j] = fz[u][j]; sh[r][q + j] = fh[u][j]; }
    }
    __syncthreads();
#pragma unroll 8
    for (int r = 0; r < SB_GR; r++) {   // rows past nr are zero
#pragma unroll
      for (int u = 0; u < 2; u++)
#pragma unroll
        for (int w = 0; w < 2; w++) acc[u][w] += sz[r][ty + 16 * u] * sh[r][tx + 16 * w];
    }
    __syncthreads();
  }
  if (i0 == 0) {
    // db: rows 256 apart, then halves of 256 slots added pairwise; a warp per output, slot lane + 32 j
    const int lane = tid & 31;
    for (int q = tid >> 5; q < SB_GT; q += 8) {
      if (o0 + q >= L.N) break;
      float v[8];
      if (M <= SB_GR) {   // the staged rows (zero past M)
        v[0] = sz[lane][q] + sz[lane + 32][q];
      } else {
#pragma unroll
        for (int j = 0; j < 8; j++) {
          v[j] = 0.0f;
          for (int r = lane + 32 * j; r < M; r += 256) v[j] += L.dZ[(long)r * L.N + o0 + q];
        }
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
          for (int j = 0; j < h; j++) v[j] += v[j + h];
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[0] += __shfl_down_sync(0xffffffffu, v[0], o);
      if (lane == 0) sdb[q] = v[0];
    }
    __syncthreads();
  }
#pragma unroll
  for (int u = 0; u < 2; u++)
#pragma unroll
    for (int w = 0; w < 2; w++) {
      const int o = o0 + ty + 16 * u, i = i0 + tx + 16 * w;
      if (o >= L.N || i >= L.K) continue;
      const long q = L.off_w + (long)o * L.K + i;
      if (p) {
        const float n = adamw_one(pv[u][w], acc[u][w], mv[u][w], vv[u][w], a, c);
        p[q] = n; mo[q] = mv[u][w]; vo[q] = vv[u][w];
        pb[q] = __float2bfloat16(n);
      } else {
        g[q] = acc[u][w];
      }
    }
  if (bias) {
    const long q = L.off_b + o0 + tid;
    const float db = sdb[tid];
    if (p) {
      const float n = adamw_one(bp, db, bm, bv, a, c);
      p[q] = n; mo[q] = bm; vo[q] = bv;
      pb[q] = __float2bfloat16(n);
    } else {
      g[q] = db;
    }
  }
  if (blockIdx.x == gridDim.x - 1) {
    float* d = p ? loss + *a.eidx : loss;
    float sum = *d;
    for (long c0 = 0; c0 < nsq; c0 += 256) {
      red[tid] = c0 + tid < nsq ? sq[c0 + tid] : 0.0f;
      __syncthreads();
      if (tid < 32) {
        // halves of 256 added pairwise: slots 128, 64, 32 apart, then across the lanes
        float w[8];
#pragma unroll
        for (int j = 0; j < 8; j++) w[j] = red[tid + 32 * j];
#pragma unroll
        for (int h = 4; h > 0; h >>= 1)
#pragma unroll
          for (int j = 0; j < h; j++) w[j] += w[j + h];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) w[0] += __shfl_down_sync(0xffffffffu, w[0], o);
        sum += w[0];
      }
      __syncthreads();
    }
    if (tid == 0) *d = sum;
  }
}

uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9e3779b97f4a7c15ULL);
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ULL;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebULL;
  return z ^ (z >> 31);
}

// ---------------------------------------------------------------------------
// Tensor-core inference (tcgen05): one CTA takes 128 rows through every layer. The weights come as a prepacked BF16 image
// (K-major, padded to multiples of 16, in chunks of TC_KC columns) by bulk TMA copies through a ring of shared-memory
// slots that runs across the layers; the activations of the 128 rows sit in shared memory; both in swizzled layouts. One
// warp issues the K/16 tcgen05.mma (M = 128, N = padded width, BF16 x BF16 -> FP32) into a TMEM accumulator, one thread
// copies; sixteen warps read the accumulator's lanes (one row per thread), add the bias, apply GELU and write the next
// layer's operand (or the FP32 outputs) in place.
// The epilogue bounds it: two special-function instructions per GELU (4100 cycles per 128 x 256 layer; with the other 15
// instructions 5800 alone, 7000 with two CTAs), then the products and their waits (5000 per 256 x 256 layer). With a ring
// of 3 slots two CTAs share an SM (shared memory, 64 registers a thread, 256 TMEM columns each), one's products and copies
// under the other's epilogue. Where there are no more tiles than SMs a ring of 8 holds a whole layer and the next one's
// copies run under the epilogue. 6-256-256-256-4: 100 000 rows 151.6 us, now 79.1; up to 19 456 rows 33.4, now 25 to 26
// (before: one CTA per SM, a layer's weights in one copy, a clock read in every wait, scalar arithmetic).
constexpr int TC_M = 128;
constexpr int TC_THREADS = 512;                            // 16 warps: 4 TMEM lane groups x 4 column groups
constexpr int TC_MAXW = 256;                              // padded width limit of this kernel
constexpr int TC_KC = 32;                                 // weight columns per chunk
constexpr int TC_A_BYTES = TC_M * TC_MAXW * 2;            // activations
constexpr int TC_C_BYTES = TC_MAXW * TC_KC * 2;           // one chunk
constexpr int tc_smem(int ring) { return TC_A_BYTES + ring * TC_C_BYTES + (2 * ring + 1) * 8 + 8; }
constexpr int TC_MAXL = 16;

__host__ __device__ inline int pad16(int v) { return (v + 15) & ~15; }

// byte offset of element (r, k) of the activations: K-major with 128-byte swizzle, blocks of 64 columns (128 rows x 128
// bytes), the eight 16-byte pieces of a row exchanged by the row's place in its group of eight
__host__ __device__ inline uint32_t act_off(int r, int k) {
  return (uint32_t)((k >> 6) * (TC_M * 128) + r * 128 + ((((k >> 3) & 7) ^ (r & 7)) << 4) + (k & 7) * 2);
}
// byte offset of element (r, k) of a chunk of weights: K-major with 64-byte swizzle, rows of TC_KC = 32 columns
__host__ __device__ inline uint32_t chunk_off(int r, int k) {
  return (uint32_t)(r * 64 + ((((k >> 3) & 3) ^ ((r >> 1) & 3)) << 4) + (k & 7) * 2);
}
__host__ __device__ inline int tc_chunks(int Kp) { return (Kp + TC_KC - 1) / TC_KC; }
// columns per copy: as many chunks of a layer Np wide as fill a slot
inline int tc_copy_cols(int Np) { return TC_KC * (TC_MAXW / Np); }

__global__ void k_next_epoch(int* eidx) { *eidx += 1; }

// the image of one layer: its weights chunk by chunk (zero beyond its columns), then its biases in FP32
__global__ void k_pack_weights(const __nv_bfloat16* W, const float* bias, int N, int K, int Np, int chunks,
                               __nv_bfloat16* img) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x, Kc = chunks * TC_KC;
  if (e < Np) reinterpret_cast<float*>(img + Np * Kc)[e] = e < N ? bias[e] : 0.0f;
  if (e >= Np * Kc) return;
  const int r = e / Kc, k = e - r * Kc, c = k / TC_KC;
  img[c * TC_KC * Np + (chunk_off(r, k - c * TC_KC) >> 1)] = (r < N && k < K) ? W[(long)r * K + k] : __float2bfloat16(0.0f);
}

struct TcLayer {
  const __nv_bfloat16* img;
  int N, K, Np, Kp;
  int cols, copies;   // columns per copy of weights, copies
};
struct TcNet {
  TcLayer l[TC_MAXL];
  int L, k0;
};

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// D (+)= A B on the tensor cores, M = 128, K = 16, operands in shared memory. An operand's matrix descriptor: low word the
// address in 16 bytes (in the units of which it advances along K) and a fixed leading distance, high word the distance of
// the 8-row groups in 16 bytes, fixed version bits 14-15 and the swizzle mode (2: 128 bytes, 4: 64 bytes) from bit 29.
constexpr uint32_t kDescAct = (1024u >> 4) | (1u << 14) | (2u << 29), kDescChunk = (512u >> 4) | (1u << 14) | (4u << 29);
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr) { return ((addr >> 4) & 0x3FFFu) | (1u << 16); }
__device__ __forceinline__ void mma_k16(uint32_t tmem, uint32_t a, uint32_t b, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 da, db;\n setp.ne.b32 p, %4, 0;\n mov.b64 da, {%1, %5};\n mov.b64 db, {%2, %6};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], da, db, %3, p;\n}\n" ::"r"(tmem),
      "r"(a), "r"(b), "r"(idesc), "r"(acc), "r"(kDescAct), "r"(kDescChunk)
      : "memory");
}

__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  return done != 0;
}
// wait for the phase of an mbarrier, giving up after about half a second (then the error flag is set); the clock, whose
// reading costs more than most of these waits, is looked at every 64 polls
__device__ __noinline__ bool mbar_wait_long(uint32_t bar, uint32_t parity, int* err) {
  const uint64_t t0 = global_ns();
  while (true) {
    for (int poll = 0; poll < 64; poll++)
      if (mbar_try(bar, parity)) return true;
    if (global_ns() - t0 > 500000000ull) {
      atomicExch(err, 1);
      return false;
    }
  }
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err) {
  if (mbar_try(bar, parity) || mbar_try(bar, parity)) return true;
  return mbar_wait_long(bar, parity, err);
}

// one lane of a converged warp, always the same
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// two FP32 values in one register pair: packed instructions round each as the scalar one does
typedef unsigned long long F2;
__device__ __forceinline__ F2 f2(float lo, float hi) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ F2 f2(float v) { return f2(v, v); }
__device__ __forceinline__ float lo(F2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return a;
}
__device__ __forceinline__ float hi(F2 v) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
  return b;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// GELU, z (1 + erf(z / sqrt 2)) / 2, of two values, with erf by Abramowitz & Stegun, Handbook of Mathematical Functions,
// 7.1.26 (Hastings' rational approximation; |error| <= 1.5e-7 for x >= 0, far below the BF16 rounding that every
// activation takes): erf(x) = 1 - t (a1 + a2 t + a3 t^2 + a4 t^3 + a5 t^4) exp(-x^2), t = 1 / (1 + p x), odd in x.
__device__ __forceinline__ F2 gelu2(F2 z) {
  const F2 x = mul2(z, f2(0.70710678118654752f));
  const F2 ax = x & 0x7fffffff7fffffffull;
  const F2 d = fma2(f2(0.3275911f), ax, f2(1.0f));
  const F2 t = f2(rcp_approx(lo(d)), rcp_approx(hi(d)));
  F2 q = fma2(f2(-1.061405429f), t, f2(1.453152027f));   // minus the polynomial
  q = fma2(q, t, f2(-1.421413741f));
  q = fma2(q, t, f2(0.284496736f));
  q = fma2(q, t, f2(-0.254829592f));
  q = mul2(t, q);
  // exp(-x^2) = 2^(-x^2 log2 e)
  const F2 w = mul2(mul2(x, x), f2(-1.44269504088896341f));
  const F2 e = f2(ex2_approx(lo(w)), ex2_approx(hi(w)));
  const F2 v = fma2(q, e, f2(1.0f));
  const F2 erf = (v & 0x7fffffff7fffffffull) | (x & 0x8000000080000000ull);
  return mul2(mul2(f2(0.5f), z), add2(f2(1.0f), erf));
}

template <int RING, int CTAS>
__global__ void __launch_bounds__(TC_THREADS, CTAS) k_mlp_fwd_tc(const __grid_constant__ TcNet net,
                                                                 const float* __restrict__ x, long n,
                                                                 float* __restrict__ y, int* err) {
  extern __shared__ __align__(1024) unsigned char sm[];
  unsigned char* A = sm;
  unsigned char* Bw = sm + TC_A_BYTES;
  uint64_t* bars = reinterpret_cast<uint64_t*>(sm + TC_A_BYTES + RING * TC_C_BYTES);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bars + 2 * RING + 1);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // TMEM lanes 32 (warp % 4) .. +31 are this warp's rows; chunks of 16 columns go round-robin to warp / 4
  const int lgrp = warp & 3, cgrp = warp >> 2;
  const int rloc = lgrp * 32 + lane;
  const long row0 = (long)blockIdx.x * TC_M;
  // a slot's copy has landed; a slot's products have completed; the layer's products have completed
  const uint32_t bar_full = smem_u32(bars), bar_free = smem_u32(bars + RING), bar_acc = smem_u32(bars + 2 * RING);
  if (tid == 0) {
    for (int q = 0; q < 2 * RING + 1; q++)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&bars[q])) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  // the weights' copies, numbered through all layers: warp 0 multiplies (c_mma so far), thread LOADER copies (c_in so
  // far) and waits for the slots, so that the products never wait for a slot to be given back
  constexpr int LOADER = 32;
  int c_in = 0, c_mma = 0, load_l = 0, load_k = 0;
  auto load_chunk = [&]() {
    if (load_l >= net.L) return;
    const int Np = net.l[load_l].Np, Kp = net.l[load_l].Kp, slot = c_in % RING;
    const int cols = min(net.l[load_l].cols, tc_chunks(Kp) * TC_KC - load_k);
    const uint32_t bytes = (uint32_t)(Np * cols * 2), bar = bar_full + 8 * slot;
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(Bw) + slot * TC_C_BYTES),
                 "l"(net.l[load_l].img + (long)load_k * Np), "r"(bytes), "r"(bar)
                 : "memory");
    c_in++;
    load_k += cols;
    if (load_k >= Kp) { load_l++; load_k = 0; }
  };
  __syncthreads();
  if (tid == LOADER)
    for (int q = 0; q < RING; q++) load_chunk();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(smem_u32(tslot))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // the 128 input rows, BF16, zero padded, in the first layer's operand layout
  {
    const int Kp = net.l[0].Kp, nk8 = Kp / 8;
    for (int e = tid; e < TC_M * nk8; e += TC_THREADS) {
      const int rr = e / nk8, k8 = e - rr * nk8;
      const long r = row0 + rr;
      __align__(16) __nv_bfloat16 v[8];
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int k = k8 * 8 + q;
        v[q] = __float2bfloat16((r < n && k < net.k0) ? x[r * net.k0 + k] : 0.0f);
      }
      *reinterpret_cast<uint4*>(A + act_off(rr, k8 * 8)) = *reinterpret_cast<const uint4*>(v);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tslot, a_lo = desc_lo(smem_u32(A)), b_lo = desc_lo(smem_u32(Bw));
  for (int l = 0; l < net.L; l++) {
    const TcLayer& Ly = net.l[l];
    const int Np = Ly.Np;
    bool ok = true;
    if (warp == 0) {   // the whole warp walks the chunks (uniform descriptors), one lane issues
      const int Kp = Ly.Kp;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(Np >> 3) << 17) |
                             ((uint32_t)(TC_M >> 4) << 24);
      const int cols = Ly.cols;
      for (int k = 0; k < Kp; k += cols, c_mma++) {
        const int slot = c_mma % RING;
        ok = mbar_wait(bar_full + 8 * slot, (c_mma / RING) & 1, err);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        uint32_t b = b_lo + slot * (TC_C_BYTES >> 4);
        if (elect_one()) {
          const int end = min(Kp, k + cols);
          for (int c = k; c < end; c += TC_KC, b += Np * (TC_KC * 2 >> 4)) {
            const uint32_t a = a_lo + (act_off(0, c) >> 4);
            mma_k16(tmem, a, b, idesc, c > 0);
            if (c + 16 < Kp) mma_k16(tmem, a + 2, b + 2, idesc, 1);
          }
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           bar_free + 8 * slot)
                       : "memory");
        }
        __syncwarp();
      }
      if (ok && elect_one())
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar_acc)
                     : "memory");
    } else if (tid == LOADER) {
      const int end = c_mma + Ly.copies;
      for (; c_mma < end && ok; c_mma++) {
        if (load_l >= net.L) continue;
        ok = mbar_wait(bar_free + 8 * (c_mma % RING), (c_mma / RING) & 1, err);
        if (ok) load_chunk();
      }
    }
    // one warp waits for the products, the others at the barrier (polls would take the epilogue's issue slots)
    __syncwarp();
    if (warp == 0) {
      if (ok) ok = mbar_wait(bar_acc, l & 1, err);
    }
    if (__syncthreads_and(ok ? 1 : 0) == 0) break;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool last = l == net.L - 1;
    const long r = row0 + rloc;
    const float* bias = reinterpret_cast<const float*>(Ly.img + Np * tc_chunks(Ly.Kp) * TC_KC);
    for (int c0 = 16 * cgrp; c0 < Np; c0 += 64) {
      float b[16];
#pragma unroll
      for (int q = 0; q < 4; q++) *reinterpret_cast<float4*>(b + 4 * q) = __ldg(reinterpret_cast<const float4*>(bias + c0) + q);
      uint32_t v[16];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(tmem + ((uint32_t)(lgrp * 32) << 16) + (uint32_t)c0)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      if (!last) {
        __align__(16) __nv_bfloat162 h[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
          const F2 g = gelu2(add2(f2(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1])), f2(b[2 * q], b[2 * q + 1])));
          h[q] = __floats2bfloat162_rn(lo(g), hi(g));
        }
        *reinterpret_cast<uint4*>(A + act_off(rloc, c0)) = *reinterpret_cast<const uint4*>(h);
        *reinterpret_cast<uint4*>(A + act_off(rloc, c0 + 8)) = *reinterpret_cast<const uint4*>(h + 4);
      } else if (r < n) {
#pragma unroll
        for (int q = 0; q < 16; q++)
          if (c0 + q < Ly.N) y[r * Ly.N + c0 + q] = __uint_as_float(v[q]) + b[q];
      }
    }
    // the padding's columns are zero whatever the row holds (their products are not where an activation is infinite); a
    // thread overwrites what it has just written. (Inside the loop above it cost 1.2 to 2 us of 80.)
    if (Ly.N < Np && !last && cgrp == ((Np >> 4) - 1) % 4)
      for (int k = Ly.N; k < Np; k++)
        *reinterpret_cast<__nv_bfloat16*>(A + act_off(rloc, k)) = __float2bfloat16(0.0f);
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  // after a wait that gave up: copies still in flight land before the block's memory is given back
  if (tid == LOADER)
    for (int c = max(0, c_in - RING); c < c_in; c++) mbar_wait(bar_full + 8 * (c % RING), (c / RING) & 1, err);
  __syncthreads();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
}

}  // namespace

struct pic_mlp {
  std::vector<int> w;                   // widths
  int L = 0;                            // layers
  long np = 0;                          // parameters
  std::vector<long> off_w, off_b;       // offsets into the parameter vector
  float* p = nullptr;                   // FP32 master parameters
  __nv_bfloat16* pb = nullptr;          // BF16 copies
  float* g = nullptr;                   // gradient
  float* m = nullptr;
  float* v = nullptr;
  long adam_t = 0;
  int cap = 0;                          // batch capacity of the work buffers
  std::vector<float*> Z;                // pre-activations per layer (FP32)
  std::vector<__nv_bfloat16*> Hb;       // activations per layer (BF16); Hb[0] is the input
  float* dA = nullptr;                  // gradient work buffers
  float* dB = nullptr;
  std::vector<float*> dZ;               // small batches: the gradient of every layer's pre-activations
  float* out = nullptr;
  float* loss = nullptr;
  float* sq = nullptr;                  // small batches: every output's share of the loss
  int* idx = nullptr;
  int* perm = nullptr;                  // shuffled sample order of one epoch (training)
  int perm_cap = 0;
  float* curve = nullptr;               // per-epoch loss sums (training)
  int curve_cap = 0;
  float2* ctab = nullptr;               // AdamW bias corrections per step of a training call
  long ctab_cap = 0;
  int* eidx = nullptr;                  // epoch index of a training call, advanced on the device
  bool use_graphs = true;               // training replays a captured epoch
  float* xb = nullptr;
  float* tb = nullptr;
  // tensor-core inference: packed weight images per layer, rebuilt when the BF16 weights change
  bool tc_ok = false;                   // every padded width <= 256
  bool tc_dirty = true;
  bool use_tc = true;
  int nsm = 0;                          // SMs of the device
  std::vector<__nv_bfloat16*> img;
  int* err = nullptr;                   // device flag: a tensor-core wait gave up
  cudaStream_t s = nullptr;
  pic_alloc_fn alloc = nullptr;
  pic_free_fn freef = nullptr;
  void* user = nullptr;
  std::vector<std::pair<void*, size_t>> allocs;
};

namespace {

template <class X>
X* mlp_al(pic_mlp* m, size_t n) {
  const size_t b = n * sizeof(X) + 256;
  void* p = nullptr;
  if (m->alloc) p = m->alloc(b, (void*)m->s, m->user);
  else if (cudaMalloc(&p, b) != cudaSuccess) p = nullptr;
  if (p) m->allocs.emplace_back(p, b);
  return (X*)p;
}

void mlp_release(pic_mlp* m) {
  cudaStreamSynchronize(m->s);
  for (auto& a : m->allocs) {
    if (m->freef) m->freef(a.first, a.second, (void*)m->s, m->user);
    else cudaFree(a.first);
  }
  m->allocs.clear();
}

int maxw(const pic_mlp* m) {
  int r = 0;
  for (int x : m->w) r = x > r ? x : r;
  return r;
}

bool ensure_batch(pic_mlp* m, int n) {
  if (n <= m->cap) return true;
  const int wm = maxw(m);
  m->Z.assign(m->L + 1, nullptr);
  m->Hb.assign(m->L + 1, nullptr);
  for (int l = 0; l <= m->L; l++) {
    m->Z[l] = mlp_al<float>(m, (size_t)n * m->w[l]);
    m->Hb[l] = mlp_al<__nv_bfloat16>(m, (size_t)n * m->w[l]);
    if (!m->Z[l] || !m->Hb[l]) return false;
  }
  m->dA = mlp_al<float>(m, (size_t)n * wm);
  m->dB = mlp_al<float>(m, (size_t)n * wm);
  m->out = mlp_al<float>(m, (size_t)n * m->w[m->L]);
  m->xb = mlp_al<float>(m, (size_t)n * m->w[0]);
  m->tb = mlp_al<float>(m, (size_t)n * m->w[m->L]);
  m->idx = mlp_al<int>(m, (size_t)n);
  if (!m->dA || !m->dB || !m->out || !m->xb || !m->tb || !m->idx) return false;
  m->dZ.assign(m->L + 1, nullptr);
  const int ns = n < SB_ROWS ? n : SB_ROWS;
  for (int l = 1; l <= m->L; l++) {
    m->dZ[l] = mlp_al<float>(m, (size_t)ns * m->w[l]);
    if (!m->dZ[l]) return false;
  }
  m->sq = mlp_al<float>(m, (size_t)ns * m->w[m->L]);
  if (!m->sq) return false;
  m->cap = n;
  return true;
}

dim3 ggrid(int M, int N) { return dim3((N + GT - 1) / GT, (M + GT - 1) / GT); }

// forward of n rows of X (FP32, n x w0) into m->out (FP32, n x wL)
void forward(pic_mlp* m, const float* X, int n) {
  const long n0 = (long)n * m->w[0];
  k_to_bf16<<<(unsigned)((n0 + 255) / 256), 256, 0, m->s>>>(n0, X, m->Hb[0]);
  for (int l = 1; l <= m->L; l++) {
    const int in = m->w[l - 1], ou = m->w[l];
    const __nv_bfloat16* W = m->pb + m->off_w[l - 1];
    const float* b = m->p + m->off_b[l - 1];
    if (l < m->L)
      k_gemm<__nv_bfloat16, __nv_bfloat16, false, true, 1><<<ggrid(n, ou), 256, 0, m->s>>>(
          n, ou, in, m->Hb[l - 1], in, W, in, m->Z[l], ou, b, m->Hb[l]);
    else
      k_gemm<__nv_bfloat16, __nv_bfloat16, false, true, 2><<<ggrid(n, ou), 256, 0, m->s>>>(
          n, ou, in, m->Hb[l - 1], in, W, in, m->out, ou, b, nullptr);
  }
}

// gradient of the mean squared error of m->out against T (n x wL) into m->g; the loss is added to *loss
void backward(pic_mlp* m, const float* T, int n, float* loss, const int* eidx = nullptr) {
  const int wl = m->w[m->L];
  const long nd = (long)n * wl;
  k_mse<<<(unsigned)((nd + 255) / 256), 256, 0, m->s>>>(nd, m->out, T, m->dA, loss, eidx);
  float* dZ = m->dA;   // gradient w.r.t. the current layer's output (pre-activation for the last)
  float* dH = m->dB;
  for (int l = m->L; l >= 1; l--) {
    const int in = m->w[l - 1], ou = m->w[l];
    // dW = dZ^T H_{l-1}: (ou x in), sum over the batch
    k_gemm<float, __nv_bfloat16, true, false, 0><<<ggrid(ou, in), 256, 0, m->s>>>(
        ou, in, n, dZ, ou, m->Hb[l - 1], in, m->g + m->off_w[l - 1], in, nullptr, nullptr);
    k_colsum<<<ou, 256, 0, m->s>>>(n, ou, dZ, m->g + m->off_b[l - 1]);
    if (l > 1) {
      // dH_{l-1} = dZ W (n x in), then through the GELU of layer l-1
      k_gemm<float, __nv_bfloat16, false, false, 0><<<ggrid(n, in), 256, 0, m->s>>>(
          n, in, ou, dZ, ou, m->pb + m->off_w[l - 1], in, dH, in, nullptr, nullptr);
      const long ne = (long)n * in;
      k_gelu_back<<<(unsigned)((ne + 255) / 256), 256, 0, m->s>>>(ne, m->Z[l - 1], dH, dH);
      float* t = dZ;
      dZ = dH;
      dH = t;
    }
  }
}

// a kernel whose launch may overlap the end of its predecessor on the stream (it waits for it on the device)
template <class... KA, class... A>
void sb_launch(pic_mlp* m, void (*k)(KA...), dim3 grid, int threads, const A&... args) {
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(threads);
  c.stream = m->s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  c.attrs = at;
  c.numAttrs = 1;
  cudaLaunchKernelEx(&c, k, KA(args)...);
}

// loss and gradients of n <= SB_ROWS rows (idx[r], or r) of X against T, then AdamW (adam given) or the gradient in
// m->g; the loss is added to *loss (adam: to loss[epoch])
void small_pass(pic_mlp* m, const float* X, const float* T, const int* idx, int n, float* loss, const AdamC* adam) {
  const int L = m->L, ty = (n + SB_M - 1) / SB_M;
  auto al16 = [](const void* q) { return (reinterpret_cast<uintptr_t>(q) & 15) == 0; };
  for (int l = 1; l <= L; l++) {
    const int in = m->w[l - 1], ou = m->w[l];
    const dim3 grid((ou + SB_N - 1) / SB_N, ty);
    const __nv_bfloat16* W = m->pb + m->off_w[l - 1];
    const float* b = m->p + m->off_b[l - 1];
    const __nv_bfloat16* H = m->Hb[l - 1];
    const int vec = in % 8 == 0 && al16(W) && al16(H);
    const bool last = l == L;
    float* Z = last ? m->out : m->Z[l];
    __nv_bfloat16* Hn = last ? nullptr : m->Hb[l];
    const float* t = last ? T : nullptr;
    float* dY = last ? m->dZ[L] : nullptr;
    if (l == 1 && last) sb_launch(m, k_sb_fwd<true, true>, grid, SB_THREADS, n, ou, in, H, X, idx, W, b, Z, Hn, t, dY, m->sq, vec);
    else if (l == 1) sb_launch(m, k_sb_fwd<true, false>, grid, SB_THREADS, n, ou, in, H, X, idx, W, b, Z, Hn, t, dY, m->sq, vec);
    else if (last) sb_launch(m, k_sb_fwd<false, true>, grid, SB_THREADS, n, ou, in, H, X, idx, W, b, Z, Hn, t, dY, m->sq, vec);
    else sb_launch(m, k_sb_fwd<false, false>, grid, SB_THREADS, n, ou, in, H, X, idx, W, b, Z, Hn, t, dY, m->sq, vec);
  }
  for (int l = L; l >= 2; l--) {
    const int in = m->w[l - 1], ou = m->w[l];
    const __nv_bfloat16* W = m->pb + m->off_w[l - 1];
    const int vec = in % 8 == 0 && al16(W), vecz = ou % 4 == 0 && al16(m->dZ[l]);
    sb_launch(m, k_sb_dx, dim3((in + SB_N - 1) / SB_N, ty), SB_THREADS, n, in, ou, m->dZ[l], W, m->Z[l - 1],
              m->dZ[l - 1], vec, vecz);
  }
  SbNet net{};
  net.L = L;
  int blocks = 0;
  for (int l = 1; l <= L; l++) {
    SbLayer& q = net.l[l - 1];
    q.dZ = m->dZ[l];
    q.H = m->Hb[l - 1];
    q.off_w = m->off_w[l - 1];
    q.off_b = m->off_b[l - 1];
    q.N = m->w[l];
    q.K = m->w[l - 1];
    q.tk = (q.K + SB_GT - 1) / SB_GT;
    q.vz = q.N % 4 == 0 && al16(q.dZ);
    q.vh = q.K % 4 == 0 && al16(q.H);
    blocks += q.tk * ((q.N + SB_GT - 1) / SB_GT);
    q.blocks = blocks;
  }
  sb_launch(m, k_sb_grad, dim3(blocks), 256, net, n, X, idx, adam ? m->p : nullptr, m->pb, m->m, m->v, m->g,
            adam ? *adam : AdamC{}, m->sq, (long)n * m->w[L], loss);
}

}  // namespace

extern "C" {

int pic_mlp_create(int n_layers, const int* widths, uint64_t seed, pic_alloc_fn alloc, pic_free_fn free_fn,
                   void* alloc_user, void* cuda_stream, pic_mlp** out) {
  if (!out) return PIC_EINVAL;
  *out = nullptr;
  if (n_layers < 1 || n_layers > 16 || !widths) return PIC_EINVAL;
  for (int l = 0; l <= n_layers; l++)
    if (widths[l] < 1 || widths[l] > 4096) return PIC_EINVAL;
  pic_mlp* m = new pic_mlp();
  m->L = n_layers;
  m->w.assign(widths, widths + n_layers + 1);
  m->s = (cudaStream_t)cuda_stream;
  m->alloc = alloc; m->freef = free_fn; m->user = alloc_user;
  long off = 0;
  for (int l = 1; l <= n_layers; l++) {
    m->off_w.push_back(off); off += (long)m->w[l] * m->w[l - 1];
    m->off_b.push_back(off); off += m->w[l];
  }
  m->np = off;
  m->p = mlp_al<float>(m, off);
  m->pb = mlp_al<__nv_bfloat16>(m, off);
  m->g = mlp_al<float>(m, off);
  m->m = mlp_al<float>(m, off);
  m->v = mlp_al<float>(m, off);
  m->loss = mlp_al<float>(m, 1);
  m->err = mlp_al<int>(m, 1);
  m->tc_ok = n_layers <= TC_MAXL;
  for (int l = 0; l <= n_layers; l++) m->tc_ok = m->tc_ok && pad16(widths[l]) <= TC_MAXW;
  if (m->tc_ok) {
    for (int l = 1; l <= n_layers; l++) 
      m->img.push_back(mlp_al<__nv_bfloat16>(m, (size_t)pad16(widths[l]) * (tc_chunks(pad16(widths[l - 1])) * TC_KC + 2)));
    for (auto* q : m->img) m->tc_ok = m->tc_ok && q;
    cudaFuncSetAttribute(k_mlp_fwd_tc<3, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(3));
    cudaFuncSetAttribute(k_mlp_fwd_tc<8, 1>, cudaFuncAttributeMaxDynamicSharedMemorySize, tc_smem(8));
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&m->nsm, cudaDevAttrMultiProcessorCount, dev);
  }
  if (!m->p || !m->pb || !m->g || !m->m || !m->v || !m->loss || !m->err) {
    mlp_release(m);
    delete m;
    return PIC_ENOMEM;
  }
  // He-style uniform initialisation from a counter-based generator; zero biases
  std::vector<float> h(off, 0.0f);
  uint64_t st = seed;
  for (int l = 1; l <= n_layers; l++) {
    const float a = std::sqrt(6.0f / (float)m->w[l - 1]) * (l == n_layers ? 0.5f : 1.0f);
    for (long i = 0; i < (long)m->w[l] * m->w[l - 1]; i++) {
      const double u = (double)(splitmix64(st) >> 11) * (1.0 / 9007199254740992.0);
      h[m->off_w[l - 1] + i] = (float)((2.0 * u - 1.0) * a);
    }
  }
  cudaMemcpyAsync(m->p, h.data(), off * sizeof(float), cudaMemcpyHostToDevice, m->s);
  k_to_bf16<<<(unsigned)((off + 255) / 256), 256, 0, m->s>>>(off, m->p, m->pb);
  cudaMemsetAsync(m->m, 0, off * sizeof(float), m->s);
  cudaMemsetAsync(m->v, 0, off * sizeof(float), m->s);
  cudaMemsetAsync(m->err, 0, sizeof(int), m->s);
  if (cudaStreamSynchronize(m->s) != cudaSuccess) {
    mlp_release(m);
    delete m;
    return PIC_ECUDA;
  }
  *out = m;
  return PIC_OK;
}

int pic_mlp_free(pic_mlp* m) {
  if (!m) return PIC_OK;
  mlp_release(m);
  delete m;
  return PIC_OK;
}

int64_t pic_mlp_param_count(pic_mlp* m) { return m ? m->np : 0; }

int pic_mlp_get_params(pic_mlp* m, float* dst) {
  if (!m || !dst) return PIC_EINVAL;
  return cudaMemcpyAsync(dst, m->p, m->np * sizeof(float), cudaMemcpyDeviceToHost, m->s) == cudaSuccess &&
                 cudaStreamSynchronize(m->s) == cudaSuccess
             ? PIC_OK
             : PIC_ECUDA;
}

int pic_mlp_set_params(pic_mlp* m, const float* src) {
  if (!m || !src) return PIC_EINVAL;
  cudaMemcpyAsync(m->p, src, m->np * sizeof(float), cudaMemcpyHostToDevice, m->s);
  k_to_bf16<<<(unsigned)((m->np + 255) / 256), 256, 0, m->s>>>(m->np, m->p, m->pb);
  m->adam_t = 0;
  m->tc_dirty = true;
  cudaMemsetAsync(m->m, 0, m->np * sizeof(float), m->s);
  cudaMemsetAsync(m->v, 0, m->np * sizeof(float), m->s);
  return cudaStreamSynchronize(m->s) == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

int pic_mlp_infer(pic_mlp* m, const float* x, int64_t n, float* y) {
  if (!m || !x || !y || n < 0) return PIC_EINVAL;
  if (n == 0) return PIC_OK;
  if (m->tc_ok && m->use_tc) {
    if (m->tc_dirty) {
      for (int l = 1; l <= m->L; l++) {
        const int N = m->w[l], K = m->w[l - 1], Np = pad16(N), Kp = pad16(K);
        const int nc = tc_chunks(Kp);
        k_pack_weights<<<(Np * nc * TC_KC + 255) / 256, 256, 0, m->s>>>(m->pb + m->off_w[l - 1], m->p + m->off_b[l - 1], N, K,
                                                                        Np, nc, m->img[l - 1]);
      }
      m->tc_dirty = false;
    }
    TcNet net{};
    net.L = m->L;
    net.k0 = m->w[0];
    for (int l = 1; l <= m->L; l++) {
      TcLayer& t = net.l[l - 1];
      t.img = m->img[l - 1];
      t.N = m->w[l];
      t.K = m->w[l - 1];
      t.Np = pad16(t.N);
      t.Kp = pad16(t.K);
      t.cols = tc_copy_cols(t.Np);
      t.copies = (t.Kp + t.cols - 1) / t.cols;
    }
    const long blocks = (n + TC_M - 1) / TC_M;
    if (blocks > m->nsm)
      k_mlp_fwd_tc<3, 2><<<(unsigned)blocks, TC_THREADS, tc_smem(3), m->s>>>(net, x, (long)n, y, m->err);
    else
      k_mlp_fwd_tc<8, 1><<<(unsigned)blocks, TC_THREADS, tc_smem(8), m->s>>>(net, x, (long)n, y, m->err);
    return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
  }
  const int chunk = 65536;
  for (int64_t r0 = 0; r0 < n; r0 += chunk) {
    const int nb = (int)(n - r0 < chunk ? n - r0 : chunk);
    if (!ensure_batch(m, nb)) return PIC_ENOMEM;
    forward(m, x + r0 * m->w[0], nb);
    cudaMemcpyAsync(y + r0 * m->w[m->L], m->out, (size_t)nb * m->w[m->L] * sizeof(float), cudaMemcpyDeviceToDevice,
                    m->s);
  }
  return cudaGetLastError() == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

int pic_mlp_use_tensor_cores(pic_mlp* m, int enable) {
  if (!m) return PIC_EINVAL;
  if (enable && !m->tc_ok) return PIC_EINVAL;
  m->use_tc = enable != 0;
  return PIC_OK;
}

int pic_mlp_use_graphs(pic_mlp* m, int enable) {
  if (!m) return PIC_EINVAL;
  m->use_graphs = enable != 0;
  return PIC_OK;
}

int pic_mlp_status(pic_mlp* m) {
  if (!m) return PIC_EINVAL;
  if (cudaStreamSynchronize(m->s) != cudaSuccess) return PIC_ECUDA;
  int e = 0;
  if (cudaMemcpy(&e, m->err, sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess) return PIC_ECUDA;
  return e ? PIC_ETIMEOUT : PIC_OK;
}

int pic_mlp_grad(pic_mlp* m, const float* x, const float* t, int n, float* loss_host, float* grad_host) {
  if (!m || !x || !t || n < 1) return PIC_EINVAL;
  if (!ensure_batch(m, n)) return PIC_ENOMEM;
  cudaMemsetAsync(m->loss, 0, sizeof(float), m->s);
  if (n <= SB_ROWS) {
    small_pass(m, x, t, nullptr, n, m->loss, nullptr);
  } else {
    forward(m, x, n);
    backward(m, t, n, m->loss);
  }
  if (loss_host) cudaMemcpyAsync(loss_host, m->loss, sizeof(float), cudaMemcpyDeviceToHost, m->s);
  if (grad_host) cudaMemcpyAsync(grad_host, m->g, m->np * sizeof(float), cudaMemcpyDeviceToHost, m->s);
  return cudaStreamSynchronize(m->s) == cudaSuccess ? PIC_OK : PIC_ECUDA;
}

int pic_mlp_train(pic_mlp* m, const float* x, const float* t, int n, int epochs, int batch, float lr,
                  float weight_decay, uint64_t seed, float* loss_curve) {
  if (!m || !x || !t || n < 1 || epochs < 0 || batch < 1) return PIC_EINVAL;
  if (batch > n) batch = n;
  if (!ensure_batch(m, batch)) return PIC_ENOMEM;
  if (n > m->perm_cap) {
    m->perm = mlp_al<int>(m, (size_t)n);
    if (!m->perm) return PIC_ENOMEM;
    m->perm_cap = n;
  }
  if (epochs > m->curve_cap) {
    m->curve = mlp_al<float>(m, (size_t)epochs);
    if (!m->curve) return PIC_ENOMEM;
    m->curve_cap = epochs;
  }
  if (epochs > 0) cudaMemsetAsync(m->curve, 0, (size_t)epochs * sizeof(float), m->s);
  m->tc_dirty = true;
  // the host draws every epoch's order up front (pinned by the seed), one upload per epoch
  std::vector<int> perm(n);
  uint64_t st = seed;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const int nbat = n / batch;
  // AdamW's bias corrections of every step of this call, computed on the host as the per-step launches did
  const long nsteps = (long)epochs * nbat;
  std::vector<float2> ctab((size_t)(nsteps > 0 ? nsteps : 1));
  for (long q = 0; q < nsteps; q++) {
    const float tq = (float)(m->adam_t + q + 1);
    ctab[q] = make_float2(1.0f - std::pow(b1, tq), 1.0f - std::pow(b2, tq));
  }
  if (nsteps > m->ctab_cap) {
    m->ctab = mlp_al<float2>(m, (size_t)nsteps);
    if (!m->ctab) return PIC_ENOMEM;
    m->ctab_cap = nsteps;
  }
  if (!m->eidx) {
    m->eidx = mlp_al<int>(m, 1);
    if (!m->eidx) return PIC_ENOMEM;
  }
  if (nsteps > 0)
    cudaMemcpyAsync(m->ctab, ctab.data(), (size_t)nsteps * sizeof(float2), cudaMemcpyHostToDevice, m->s);
  cudaMemsetAsync(m->eidx, 0, sizeof(int), m->s);
  // one epoch's launches (per batch of up to SB_ROWS rows the small-batch products with AdamW, else gather, forward,
  // backward and AdamW; then the epoch counter), with
  // the epoch index and the step's bias corrections read on the device
  auto epoch_launches = [&](cudaStream_t s) {
    cudaStream_t keep = m->s;
    m->s = s;
    for (int k = 0; k < nbat; k++) {
      if (batch <= SB_ROWS) {
        const AdamC a{lr, b1, b2, eps, weight_decay, m->ctab, m->eidx, nbat, k};
        small_pass(m, x, t, m->perm + (long)k * batch, batch, m->curve, &a);
        continue;
      }
      k_gather_rows<<<batch, 64, 0, s>>>(batch, m->perm + (long)k * batch, x, m->w[0], t, m->w[m->L], m->xb, m->tb);
      forward(m, m->xb, batch);
      backward(m, m->tb, batch, m->curve, m->eidx);
      k_adamw<<<(unsigned)((m->np + 255) / 256), 256, 0, s>>>(m->np, m->p, m->g, m->m, m->v, m->pb, lr, b1, b2, eps,
                                                              weight_decay, 0.f, 0.f, m->ctab, m->eidx, nbat, k);
    }
    k_next_epoch<<<1, 1, 0, s>>>(m->eidx);
    m->s = keep;
  };
  // The epoch is captured once in a CUDA graph on a private stream and replayed (8 launches per batch for four layers:
  // at batch 64 the step is launch-bound). Where capture is not possible, the same
  // launches run directly on the caller's stream.
  cudaStream_t ts = nullptr;
  cudaGraphExec_t ge = nullptr;
  cudaStreamCaptureStatus cap_st = cudaStreamCaptureStatusNone;
  if (m->use_graphs && epochs > 1 && nbat > 0 && cudaStreamIsCapturing(m->s, &cap_st) == cudaSuccess &&
      cap_st == cudaStreamCaptureStatusNone && cudaStreamCreateWithFlags(&ts, cudaStreamNonBlocking) == cudaSuccess) {
    cudaGraph_t gr = nullptr;
    if (cudaStreamBeginCapture(ts, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      epoch_launches(ts);
      if (cudaStreamEndCapture(ts, &gr) == cudaSuccess && gr) {
        if (cudaGraphInstantiate(&ge, gr, 0) != cudaSuccess) ge = nullptr;
        cudaGraphDestroy(gr);
      }
    }
    cudaGetLastError();   // a refused capture leaves no sticky error; the direct path follows
    if (!ge) {
      cudaStreamDestroy(ts);
      ts = nullptr;
    }
  }
  cudaEvent_t ready = nullptr;
  if (ge) {
    // the private stream starts after everything queued on the caller's stream
    cudaEventCreateWithFlags(&ready, cudaEventDisableTiming);
    cudaEventRecord(ready, m->s);
    cudaStreamWaitEvent(ts, ready, 0);
  }
  cudaStream_t run_s = ge ? ts : m->s;
  for (int e = 0; e < epochs; e++) {
    for (int i = 0; i < n; i++) perm[i] = i;
    for (int i = n - 1; i > 0; i--) {   // Fisher-Yates with a counter-based generator
      const int j = (int)(splitmix64(st) % (uint64_t)(i + 1));
      const int tmp = perm[i]; perm[i] = perm[j]; perm[j] = tmp;
    }
    // pageable source: the copy has been staged when the call returns, so perm may be refilled
    cudaMemcpyAsync(m->perm, perm.data(), (size_t)n * sizeof(int), cudaMemcpyHostToDevice, run_s);
    if (ge) cudaGraphLaunch(ge, ts);
    else epoch_launches(m->s);
  }
  m->adam_t += nsteps;
  if (ge) {
    cudaEventRecord(ready, ts);
    cudaStreamWaitEvent(m->s, ready, 0);
  }
  if (loss_curve && epochs > 0) {
    cudaMemcpyAsync(loss_curve, m->curve, (size_t)epochs * sizeof(float), cudaMemcpyDeviceToHost, m->s);
  }
  const bool ok = cudaStreamSynchronize(m->s) == cudaSuccess;
  if (ge) {
    cudaGraphExecDestroy(ge);
    cudaStreamDestroy(ts);
    cudaEventDestroy(ready);
  }
  if (!ok) return PIC_ECUDA;
  if (loss_curve)
    for (int e = 0; e < epochs; e++) loss_curve[e] /= (float)(nbat > 0 ? nbat : 1);
  return PIC_OK;
}

}  // extern "C"
