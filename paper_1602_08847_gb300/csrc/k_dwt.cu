// W_s as a union of eight orthonormal Daubechies wavelet bases, the
// comparison dictionary of Sec. 4 (the one of the first MUFFIN version):
//   W_s x = (1/sqrt 8) [Psi_1 x; ...; Psi_8 x],
// Psi_p the J-level periodic separable 2D discrete wavelet transform with the
// Daubechies filter of p vanishing moments, coefficients of each basis in the
// Mallat layout of an N x N plane (level j transforms the top-left
// (N/2^j)^2 square; its detail quadrants are final, its low-low quadrant feeds
// level j+1).  W_s^T W_s = I (a tight frame).
//
// One analysis step along an axis of even length M:
//   lo[k] = sum_t h[t] x[(2k + t) mod M],  hi[k] = sum_t g[t] x[(2k + t) mod M],
//   g[t] = (-1)^t h[2p-1-t];
// its adjoint (= inverse, the bank is orthonormal):
//   x[i] = sum_{t = i mod 2} h[t] lo[k] + g[t] hi[k],  k = ((i - t) mod M) / 2.
// Every launch covers all channels and all eight bases.  One kernel per level
// and direction: a block owns a group of rows over the full width, filters
// them along one axis into shared memory and from there along the other, each
// thread a run of outputs with its inputs in registers, so that a value read
// feeds several multiply-adds (compile-time filter length, taps as constant
// operands).  The finest level of the adjoint runs the eight bases one after
// another in a block and sums them in registers, so the per-basis images are
// never stored.  Levels below 32 x 32 take small kernels that read straight
// from global memory.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <complex>
#include <vector>

#include "device.cuh"
#include "internal.h"

namespace muffin {

constexpr int kMaxTaps = 16;

__constant__ float c_dbh[kDbBases][kMaxTaps];
__constant__ float c_dbg[kDbBases][kMaxTaps];

// ------------------------------------------------------------------ filters (host)

// H(z) = sqrt(2) ((1 + z^-1)/2)^p Q(z) with |Q(e^iw)|^2 = P(sin^2(w/2)),
// P(y) = sum_{k<p} C(p-1+k, k) y^k; each root y_k of P gives the pair of
// z roots of z^2 - 2(1 - 2y_k) z + 1, of which Q keeps the one inside the unit
// circle (minimum phase); Q(1) = 1.  Roots of P by the Weierstrass
// (Durand-Kerner) iteration.
bool daubechies_lowpass(int p, double* h) {
  using cd = std::complex<double>;
  if (p < 1 || p > kDbBases || !h) return false;
  const int deg = p - 1;
  std::vector<double> a(p);   // ascending coefficients of P
  for (int k = 0; k < p; ++k) {
    double c = 1.0;           // C(p-1+k, k)
    for (int i = 1; i <= k; ++i) c = c * (p - 1 + i) / i;
    a[k] = c;
  }
  std::vector<cd> roots(deg);
  if (deg > 0) {
    auto eval = [&](cd y) {   // monic P(y) / a[deg]
      cd v = 1.0;
      for (int k = deg - 1; k >= 0; --k) v = v * y + a[k] / a[deg];
      return v;
    };
    const cd seed(0.4, 0.9);
    cd w = 1.0;
    for (int i = 0; i < deg; ++i) { roots[i] = w; w *= seed; }
    for (int it = 0; it < 2000; ++it) {
      double move = 0.0;
      for (int i = 0; i < deg; ++i) {
        cd den = 1.0;
        for (int j = 0; j < deg; ++j) if (j != i) den *= roots[i] - roots[j];
        const cd d = eval(roots[i]) / den;
        roots[i] -= d;
        move = std::max(move, std::abs(d));
      }
      if (move < 1e-16) break;
    }
  }
  std::vector<cd> q(1, cd(1.0));
  for (int i = 0; i < deg; ++i) {
    const cd aa = 1.0 - 2.0 * roots[i];
    const cd r = std::sqrt(aa * aa - 1.0);
    const cd zk = std::abs(aa + r) < 1.0 ? aa + r : aa - r;
    std::vector<cd> nq(q.size() + 1, cd(0.0));
    for (size_t t = 0; t < q.size(); ++t) { nq[t] += q[t]; nq[t + 1] -= zk * q[t]; }
    for (auto& v : nq) v /= (1.0 - zk);
    q.swap(nq);
  }
  std::vector<double> binom(p + 1);
  for (int t = 0; t <= p; ++t) {
    double c = 1.0;
    for (int i = 1; i <= t; ++i) c = c * (p - t + i) / i;
    binom[t] = c / std::ldexp(1.0, p);
  }
  for (int t = 0; t < 2 * p; ++t) {
    cd acc = 0.0;
    for (int u = 0; u <= p; ++u) {
      const int v = t - u;
      if (v >= 0 && v < (int)q.size()) acc += binom[u] * q[v];
    }
    h[t] = std::sqrt(2.0) * acc.real();
  }
  return true;
}

// ------------------------------------------------------------------ kernels

constexpr float kUnionScale = 0.35355339059327373f;   // 1/sqrt(8)
constexpr int kRowsPerBlock = 8;
constexpr int kMinTile = 32;      // smallest level of the row-group kernels

// The kernels below run one body per basis, instantiated for its filter length
// (TAPS = 2p, compile time) so that every tap loop unrolls and its loads issue
// together; the block's basis b = blockIdx.z & 7 picks the body.
#define MUFFIN_DB_DISPATCH(CALL) \
  switch (blockIdx.z & 7) {      \
    case 0: CALL(2); break;      \
    case 1: CALL(4); break;      \
    case 2: CALL(6); break;      \
    case 3: CALL(8); break;      \
    case 4: CALL(10); break;     \
    case 5: CALL(12); break;     \
    case 6: CALL(14); break;     \
    default: CALL(16); break;    \
  }

// ------------------------------------------------------------------ row-group kernels, levels of at least 32 x 32
//
// 256 x 256 x 64, four levels, us per pass: analysis 258 -> 157, adjoint 399 ->
// 117, bitwise the same (before: a thread per output, one load for every one or
// two multiply-adds, and for the adjoint columns and rows in separate kernels
// with the images between them in global memory).  The analysis is bound by the
// L1 reads of its row filter and the read-modify-write of U (40 us of DRAM at
// copy speed), the adjoint by the FP32 pipe at 16 warps per SM.

// Analysis of level M: rows q0 .. q0 + Q - 1 of the low and of the high half,
// from the input rows 2 q0 .. 2 q0 + 2Q + TAPS - 3.  Shared: those rows after
// the row filter, [row][M] (low columns, then high ones).
template <int MODE, int TAPS, int Q>
__device__ __forceinline__ void dwt_rows_body(const float* __restrict__ src, float* __restrict__ ll,
                                              float* __restrict__ U, int n, int M, int last, float kk, float rho,
                                              float* __restrict__ sY) {
  constexpr int b = TAPS / 2 - 1, ROWS = 2 * Q + TAPS - 2, NV = (8 + TAPS - 2 + 3) / 4;
  const int H = M >> 1, m = M - 1, q0 = blockIdx.x * Q;
  // rows: an item is four low and four high outputs of a row, from 8 + TAPS - 2 inputs
  const int runs = M >> 3;
  for (int it = threadIdx.x; it < ROWS * runs; it += blockDim.x) {
    const int r = it / runs, k0 = 4 * (it - r * runs);
    const float* row = src + (size_t)((2 * q0 + r) & m) * n;
    float x[4 * NV];
#pragma unroll
    for (int v = 0; v < NV; ++v) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(row + ((2 * k0 + 4 * v) & m)));
      x[4 * v] = t.x; x[4 * v + 1] = t.y; x[4 * v + 2] = t.z; x[4 * v + 3] = t.w;
    }
    float lo[4] = {}, hi[4] = {};
#pragma unroll
    for (int t = 0; t < TAPS; ++t)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        lo[e] = fmaf(c_dbh[b][t], x[2 * e + t], lo[e]);
        hi[e] = fmaf(c_dbg[b][t], x[2 * e + t], hi[e]);
      }
    *reinterpret_cast<float4*>(sY + r * M + k0) = make_float4(lo[0], lo[1], lo[2], lo[3]);
    *reinterpret_cast<float4*>(sY + r * M + H + k0) = make_float4(hi[0], hi[1], hi[2], hi[3]);
  }
  __syncthreads();
  for (int c = threadIdx.x; c < M; c += blockDim.x) {
    const bool keep = c < H && !last;            // the low-low quadrant feeds the next level
    float* ul = U + (size_t)q0 * n + c;
    float* uh = ul + (size_t)H * n;
    float ol[Q], oh[Q];                           // old duals, loaded under the column filter
    if (MODE == MODE_UPDATE) {
#pragma unroll
      for (int q = 0; q < Q; ++q) {
        ol[q] = keep ? 0.f : ul[(size_t)q * n];
        oh[q] = uh[(size_t)q * n];
      }
    }
    float x[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) x[r] = sY[r * M + c];
    auto dual = [&](float o, float w) {
      w *= kUnionScale;
      return MODE == MODE_UPDATE ? rho * sat1(o + kk * w) + (1.0f - rho) * o : w;
    };
#pragma unroll
    for (int q = 0; q < Q; ++q) {
      float lo = 0.f, hi = 0.f;
#pragma unroll
      for (int t = 0; t < TAPS; ++t) {
        lo = fmaf(c_dbh[b][t], x[2 * q + t], lo);
        hi = fmaf(c_dbg[b][t], x[2 * q + t], hi);
      }
      if (keep) ll[(size_t)(q0 + q) * n + c] = lo;
      else ul[(size_t)q * n] = dual(ol[q], lo);
      uh[(size_t)q * n] = dual(oh[q], hi);
    }
  }
}

// grid (M / 2 / Q, 1, 8 L); shared (2Q + 14) M floats
template <int MODE, int Q>
__global__ void __launch_bounds__(512)
k_dwt_rows(const float* __restrict__ src0, const float* __restrict__ llin, float* __restrict__ ll,
           float* __restrict__ U, int n, int M, int level0, int last, float kk, float rho) {
  extern __shared__ __align__(16) float sY[];
  const size_t P = (size_t)n * n;
  const int z = blockIdx.z;
  const float* src = level0 ? src0 + (size_t)(z >> 3) * P : llin + (size_t)z * P;
#define CALL(T) dwt_rows_body<MODE, T, Q>(src, ll + (size_t)z * P, U + (size_t)z * P, n, M, last, kk, rho, sY)
  MUFFIN_DB_DISPATCH(CALL)
#undef CALL
}

// Shared slot of column x: four spare floats after every 32, so that the
// 16-byte reads of lanes 32 bytes apart fall into different banks.
__device__ __forceinline__ int syn_slot(int x) { return x + ((x >> 5) << 2); }
__host__ __device__ constexpr int syn_pitch(int M) { return M + M / 8; }

// Adjoint of one basis and level M for output rows 2 q0 .. 2 q0 + R - 1: adds
// this thread's 16 outputs (row, 16 columns from 16 run) to acc.  lo / hi of
// column c: rows of the low-low image (c < H, unless this is the coarsest
// level) or of U, and rows H .. of U.  Shared: [R][syn_pitch(M)].
template <int TAPS, int R>
__device__ __forceinline__ void idwt_group(const float* __restrict__ U, const float* __restrict__ llin, int n, int M,
                                           int q0, int coarsest, float* __restrict__ sV, int row, int run,
                                           float (&acc)[16]) {
  constexpr int b = TAPS / 2 - 1, p = TAPS / 2, NQ = R / 2, NW = (p - 1 + 3) / 4;   // NW chunks before the run
  const int H = M >> 1, hm = H - 1, pitch = syn_pitch(M);
  for (int c = threadIdx.x; c < M; c += blockDim.x) {
    const float* lo = (c < H && !coarsest ? llin : U) + c;
    const float* hi = U + (size_t)H * n + c;
    float a[NQ + p - 1], d[NQ + p - 1];
#pragma unroll
    for (int i = 0; i < NQ + p - 1; ++i) {
      const size_t k = (size_t)((q0 - (p - 1) + i) & hm) * n;
      a[i] = __ldg(lo + k);
      d[i] = __ldg(hi + k);
    }
#pragma unroll
    for (int q = 0; q < NQ; ++q)
#pragma unroll
      for (int par = 0; par < 2; ++par) {
        float v = 0.f;
#pragma unroll
        for (int s = 0; s < p; ++s) {
          v = fmaf(c_dbh[b][par + 2 * s], a[q + p - 1 - s], v);
          v = fmaf(c_dbg[b][par + 2 * s], d[q + p - 1 - s], v);
        }
        sV[(2 * q + par) * pitch + syn_slot(c)] = v;
      }
  }
  __syncthreads();
  const float* vr = sV + row * pitch;
  const int u0 = 8 * run;
  float a[4 * NW + 8], d[4 * NW + 8];
#pragma unroll
  for (int i = 0; i < NW + 2; ++i) {
    const int u = (u0 - 4 * NW + 4 * i) & hm;
    const float4 x = *reinterpret_cast<const float4*>(vr + syn_slot(u));
    const float4 y = *reinterpret_cast<const float4*>(vr + syn_slot(H + u));
    a[4 * i] = x.x; a[4 * i + 1] = x.y; a[4 * i + 2] = x.z; a[4 * i + 3] = x.w;
    d[4 * i] = y.x; d[4 * i + 1] = y.y; d[4 * i + 2] = y.z; d[4 * i + 3] = y.w;
  }
#pragma unroll
  for (int e = 0; e < 8; ++e)
#pragma unroll
    for (int par = 0; par < 2; ++par) {
      float v = 0.f;
#pragma unroll
      for (int s = 0; s < p; ++s) {
        v = fmaf(c_dbh[b][par + 2 * s], a[4 * NW + e - s], v);
        v = fmaf(c_dbg[b][par + 2 * s], d[4 * NW + e - s], v);
      }
      acc[2 * e + par] += v;
    }
  __syncthreads();       // the next basis overwrites sV
}

__device__ __forceinline__ void put16(float* __restrict__ o, const float (&v)[16], float k) {
#pragma unroll
  for (int i = 0; i < 4; ++i)
    reinterpret_cast<float4*>(o)[i] = make_float4(k * v[4 * i], k * v[4 * i + 1], k * v[4 * i + 2], k * v[4 * i + 3]);
}

// One level and basis: grid (M / R, 1, 8 L), M R / 16 threads.
template <int R>
__global__ void __launch_bounds__(512)
k_idwt_group(const float* __restrict__ U, const float* __restrict__ llin, float* __restrict__ out, int n, int M,
             int coarsest) {
  extern __shared__ __align__(16) float sV[];
  const size_t z = blockIdx.z, P = (size_t)n * n;
  const int row = threadIdx.x / (M >> 4), run = threadIdx.x % (M >> 4);
  float acc[16] = {};
#define CALL(T) idwt_group<T, R>(U + z * P, llin + z * P, n, M, blockIdx.x * (R / 2), coarsest, sV, row, run, acc)
  MUFFIN_DB_DISPATCH(CALL)
#undef CALL
  put16(out + z * P + (size_t)(blockIdx.x * R + row) * n + 16 * run, acc, 1.0f);
}

// Finest level, all eight bases: S = (1/sqrt 8) sum_b.  grid (N / R, 1, L).
template <int R>
__global__ void __launch_bounds__(512)
k_idwt_group_sum(const float* __restrict__ U, const float* __restrict__ llin, float* __restrict__ S, int n,
                 int coarsest) {
  extern __shared__ __align__(16) float sV[];
  const size_t l = blockIdx.z, P = (size_t)n * n;
  const int row = threadIdx.x / (n >> 4), run = threadIdx.x % (n >> 4), q0 = blockIdx.x * (R / 2);
  const float *u = U + l * kDbBases * P, *w = llin + l * kDbBases * P;
  float acc[16] = {};
  idwt_group<2, R>(u, w, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<4, R>(u + P, w + P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<6, R>(u + 2 * P, w + 2 * P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<8, R>(u + 3 * P, w + 3 * P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<10, R>(u + 4 * P, w + 4 * P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<12, R>(u + 5 * P, w + 5 * P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<14, R>(u + 6 * P, w + 6 * P, n, n, q0, coarsest, sV, row, run, acc);
  idwt_group<16, R>(u + 7 * P, w + 7 * P, n, n, q0, coarsest, sV, row, run, acc);
  put16(S + l * P + (size_t)(blockIdx.x * R + row) * n + 16 * run, acc, kUnionScale);
}

// ------------------------------------------------------------------ small levels, at most 16 x 16

// Analysis of one whole level of at most 16 x 16, rows and columns fused through
// shared memory.  A block owns the low or the high half of the columns of the
// row-transformed plane: it computes them for all M rows into shared memory (row
// filter, inputs read through L1), then filters each of its columns: the low-low
// quadrant feeds the next level (written to `ll`, which the caller alternates
// between two scratch planes so that no level overwrites the plane it reads),
// every final coefficient updates U.  grid (2, 1, 8 L), shared memory M H floats.
template <int MODE, int TAPS>
__device__ __forceinline__ void dwt_level_body(const float* __restrict__ src0, const float* __restrict__ llin,
                                               float* __restrict__ ll, float* __restrict__ U, int n, int M,
                                               int level0, int last, float kk, float rho, float* __restrict__ sY) {
  const int z = blockIdx.z, b = z & 7, l = z >> 3;
  const int H = M >> 1, m = M - 1;
  const size_t P = (size_t)n * n;
  const bool hic = blockIdx.x == 1;            // the high-pass (detail) columns
  const float* src = level0 ? src0 + (size_t)l * P : llin + (size_t)z * P;
  const int lsc = __ffs(H) - 1;
  // the basis' filters in registers (constant-memory reads per tap would cost an issue slot each)
  float hf[TAPS], gf[TAPS];
#pragma unroll
  for (int t = 0; t < TAPS; ++t) {
    hf[t] = c_dbh[b][t];
    gf[t] = c_dbg[b][t];
  }
  for (int idx = threadIdx.x; idx < M * H; idx += blockDim.x) {
    const int r = idx >> lsc, j = idx & (H - 1);
    const float* row = src + (size_t)r * n;
    const int base = 2 * j;
    // taps in aligned pairs: (2k + t) is even for even t and M is even, so x[t + 1] follows x[t]
    float x[TAPS];
#pragma unroll
    for (int t = 0; t < TAPS; t += 2) {
      const float2 v = __ldg(reinterpret_cast<const float2*>(row + ((base + t) & m)));
      x[t] = v.x;
      x[t + 1] = v.y;
    }
    float acc = 0.f;
#pragma unroll
    for (int t = 0; t < TAPS; ++t) acc = fmaf(hic ? gf[t] : hf[t], x[t], acc);
    sY[idx] = acc;
  }
  __syncthreads();
  float* Uz = U + (size_t)z * P;
  auto put = [&](int row, int c, float w) {
    float* u = Uz + (size_t)row * n + c;
    w *= kUnionScale;
    if (MODE == MODE_UPDATE) {
      const float uo = *u;
      *u = rho * sat1(uo + kk * w) + (1.0f - rho) * uo;
    } else {
      *u = w;
    }
  };
  for (int idx = threadIdx.x; idx < H * H; idx += blockDim.x) {
    const int q = idx >> lsc, j = idx & (H - 1), c = hic ? H + j : j;
    float x[TAPS];
#pragma unroll
    for (int t = 0; t < TAPS; ++t) x[t] = sY[(((2 * q + t) & m) << lsc) + j];
    float lo = 0.f, hi = 0.f;
#pragma unroll
    for (int t = 0; t < TAPS; ++t) {
      lo = fmaf(hf[t], x[t], lo);
      hi = fmaf(gf[t], x[t], hi);
    }
    if (!hic && !last) ll[(size_t)z * P + (size_t)q * n + c] = lo;
    else put(q, c, lo);
    put(H + q, c, hi);
  }
}

template <int MODE>
__global__ void __launch_bounds__(128)
k_dwt_level(const float* __restrict__ src0, const float* __restrict__ llin, float* __restrict__ ll,
            float* __restrict__ U, int n, int M, int level0, int last, float kk, float rho) {
  extern __shared__ float sY[];
#define CALL(T) dwt_level_body<MODE, T>(src0, llin, ll, U, n, M, level0, last, kk, rho, sY)
  MUFFIN_DB_DISPATCH(CALL)
#undef CALL
}

// Adjoint, columns of level M: W1[z][i][c] from the low half (rows < M/2:
// the low-low quadrant from W2[z], or from U at the coarsest level, next to the
// U quadrant for c >= M/2) and the high half (U rows >= M/2).
template <int TAPS>
__device__ __forceinline__ void idwt_cols_body(const float* __restrict__ U, const float* __restrict__ W2,
                                               float* __restrict__ W1, int n, int M, int coarsest) {
  const int z = blockIdx.z, b = z & 7;
  const int c = threadIdx.x;
  const int H = M >> 1, m = M - 1;
  if (c >= M) return;
  const size_t P = (size_t)n * n;
  const float* lo = ((c < H && !coarsest) ? W2 : U) + (size_t)z * P + c;
  const float* hi = U + (size_t)z * P + (size_t)H * n + c;
  // output rows i of this thread all have the parity of threadIdx.y (blockDim.y is even): its taps in registers
  const int par = threadIdx.y & 1;
  float he[TAPS / 2], ge[TAPS / 2];
#pragma unroll
  for (int s2 = 0; s2 < TAPS / 2; ++s2) {
    he[s2] = c_dbh[b][par + 2 * s2];
    ge[s2] = c_dbg[b][par + 2 * s2];
  }
#pragma unroll 1
  for (int i = threadIdx.y; i < M; i += blockDim.y) {
    float a[TAPS / 2], d[TAPS / 2];
#pragma unroll
    for (int s2 = 0; s2 < TAPS / 2; ++s2) {
      const size_t kk = (size_t)(((i - par - 2 * s2) & m) >> 1) * n;
      a[s2] = __ldg(lo + kk);
      d[s2] = __ldg(hi + kk);
    }
    float acc = 0.f;
#pragma unroll
    for (int s2 = 0; s2 < TAPS / 2; ++s2) {
      acc = fmaf(he[s2], a[s2], acc);
      acc = fmaf(ge[s2], d[s2], acc);
    }
    W1[(size_t)z * P + (size_t)i * n + c] = acc;
  }
}

__global__ void k_idwt_cols(const float* __restrict__ U, const float* __restrict__ W2, float* __restrict__ W1,
                            int n, int M, int coarsest) {
#define CALL(T) idwt_cols_body<T>(U, W2, W1, n, M, coarsest)
  MUFFIN_DB_DISPATCH(CALL)
#undef CALL
}

// Adjoint, rows of level M: out[z][r][i] from W1[z][r][k] (low) and W1[z][r][M/2 + k] (high).
// The first half of the block computes the even outputs i = 2u, the second
// half the odd ones, so that each thread's taps sit in registers and the
// loads of a warp are consecutive.
template <int TAPS>
__device__ __forceinline__ void idwt_rows_body(const float* __restrict__ W1, float* __restrict__ out, int n, int M) {
  const int z = blockIdx.z, b = z & 7;
  const int H = M >> 1;
  const size_t P = (size_t)n * n;
  const int half = blockDim.x >> 1, par = threadIdx.x >= half, u0 = threadIdx.x - par * half;
  float he[TAPS / 2], ge[TAPS / 2];
#pragma unroll
  for (int s2 = 0; s2 < TAPS / 2; ++s2) {
    he[s2] = c_dbh[b][par + 2 * s2];
    ge[s2] = c_dbg[b][par + 2 * s2];
  }
  const int r1 = min(M, (int)(blockIdx.y + 1) * kRowsPerBlock);
  for (int r = blockIdx.y * kRowsPerBlock; r < r1; ++r) {
    const float* src = W1 + (size_t)z * P + (size_t)r * n;
    float* dst = out + (size_t)z * P + (size_t)r * n;
    for (int u = u0; u < H; u += half) {
      float a[TAPS / 2], d[TAPS / 2];
#pragma unroll
      for (int s2 = 0; s2 < TAPS / 2; ++s2) {
        const int kk = (u - s2) & (H - 1);   // ((2u + par - par - 2 s2) mod M) / 2
        a[s2] = __ldg(src + kk);
        d[s2] = __ldg(src + H + kk);
      }
      float acc = 0.f;
#pragma unroll
      for (int s2 = 0; s2 < TAPS / 2; ++s2) {
        acc = fmaf(he[s2], a[s2], acc);
        acc = fmaf(ge[s2], d[s2], acc);
      }
      dst[2 * u + par] = acc;
    }
  }
}

__global__ void k_idwt_rows(const float* __restrict__ W1, float* __restrict__ out, int n, int M) {
#define CALL(T) idwt_rows_body<T>(W1, out, n, M)
  MUFFIN_DB_DISPATCH(CALL)
#undef CALL
}

// Finest level of the adjoint, rows, for all eight bases at once: S[l][r][i] =
// (1/sqrt 8) sum_b (row synthesis of W1[l][b] at (r, i)), bases summed in
// order, so the per-basis images are never stored.  grid (1, row groups, L).
template <int TAPS>
__device__ __forceinline__ float idwt_row_value(const float* __restrict__ src, int b, int u, int par, int H) {
  float a[TAPS / 2], d[TAPS / 2];
#pragma unroll
  for (int s2 = 0; s2 < TAPS / 2; ++s2) {
    const int kk = (u - s2) & (H - 1);
    a[s2] = __ldg(src + kk);
    d[s2] = __ldg(src + H + kk);
  }
  float acc = 0.f;
#pragma unroll
  for (int s2 = 0; s2 < TAPS / 2; ++s2) {
    acc = fmaf(c_dbh[b][par + 2 * s2], a[s2], acc);   // par is the same across a warp: one broadcast read
    acc = fmaf(c_dbg[b][par + 2 * s2], d[s2], acc);
  }
  return acc;
}

// Output i = 2u + par: the first half of the block takes the even outputs, the second the odd ones.
__global__ void k_idwt_rows_sum(const float* __restrict__ W1, float* __restrict__ S, int n) {
  const int l = blockIdx.z, M = n, H = M >> 1;
  const size_t P = (size_t)n * n;
  const int half = blockDim.x >> 1, par = threadIdx.x >= half, u0 = threadIdx.x - par * half;
  const int r1 = min(M, (int)(blockIdx.y + 1) * kRowsPerBlock);
  for (int r = blockIdx.y * kRowsPerBlock; r < r1; ++r) {
    const float* src = W1 + (size_t)l * kDbBases * P + (size_t)r * n;
    for (int u = u0; u < H; u += half) {
      float acc = idwt_row_value<2>(src, 0, u, par, H);
      acc += idwt_row_value<4>(src + P, 1, u, par, H);
      acc += idwt_row_value<6>(src + 2 * P, 2, u, par, H);
      acc += idwt_row_value<8>(src + 3 * P, 3, u, par, H);
      acc += idwt_row_value<10>(src + 4 * P, 4, u, par, H);
      acc += idwt_row_value<12>(src + 5 * P, 5, u, par, H);
      acc += idwt_row_value<14>(src + 6 * P, 6, u, par, H);
      acc += idwt_row_value<16>(src + 7 * P, 7, u, par, H);
      S[(size_t)l * P + (size_t)r * n + 2 * u + par] = kUnionScale * acc;
    }
  }
}

__global__ void k_abs_sum(const float* __restrict__ x, size_t n, double* __restrict__ partials) {
  __shared__ double red[32];
  double acc = 0.0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    acc += fabs((double)x[i]);
  const double t = block_sum(acc, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = t;
}

cudaError_t dwt_configure() {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static bool done[64] = {};
  if (dev < 64 && done[dev]) return cudaSuccess;
  float hf[kDbBases][kMaxTaps] = {}, gf[kDbBases][kMaxTaps] = {};
  for (int b = 0; b < kDbBases; ++b) {
    double h[kMaxTaps];
    const int p = b + 1, taps = 2 * p;
    daubechies_lowpass(p, h);
    for (int t = 0; t < taps; ++t) {
      hf[b][t] = (float)h[t];
      gf[b][t] = (float)((t & 1 ? -1.0 : 1.0) * h[taps - 1 - t]);
    }
  }
  if ((e = cudaMemcpyToSymbol(c_dbh, hf, sizeof(hf))) != cudaSuccess) return e;
  if ((e = cudaMemcpyToSymbol(c_dbg, gf, sizeof(gf))) != cudaSuccess) return e;
  if ((e = allow_max_dyn_smem(k_dwt_rows<MODE_UPDATE, 8>)) != cudaSuccess) return e;
  if ((e = allow_max_dyn_smem(k_dwt_rows<MODE_LINEAR, 8>)) != cudaSuccess) return e;
  if ((e = allow_max_dyn_smem(k_idwt_group<16>)) != cudaSuccess) return e;
  if ((e = allow_max_dyn_smem(k_idwt_group_sum<16>)) != cudaSuccess) return e;
  if ((e = allow_max_dyn_smem(k_idwt_group_sum<8>)) != cudaSuccess) return e;
  if (dev < 64) done[dev] = true;
  return cudaSuccess;
}

// ------------------------------------------------------------------ launchers

template <int MODE>
static void dwt_level(const Geom& g, const DwtArgs& a, int j, cudaStream_t s) {
  const int n = g.n, Z = kDbBases * g.L, M = n >> j, last = j == g.J - 1;
  // level j reads the low-low plane level j - 1 wrote and writes its own to the other scratch plane
  const float* llin = (j & 1) ? a.W1 : a.W2;
  float* ll = (j & 1) ? a.W2 : a.W1;
  const float kk = MODE == MODE_UPDATE ? a.k : 1.f, rho = MODE == MODE_UPDATE ? a.rho : 1.f;
  if (M >= kMinTile) {
    // eight output rows of each half a block (their 16 + TAPS - 2 input rows overlap the next block's by TAPS - 2)
    constexpr int Q = 8;
    k_dwt_rows<MODE, Q><<<dim3(M / 2 / Q, 1, Z), M < 512 ? M : 512, (size_t)(2 * Q + kMaxTaps - 2) * M * sizeof(float), s>>>(
        a.src, llin, ll, a.U, n, M, j == 0, last, kk, rho);
  } else {
    k_dwt_level<MODE><<<dim3(2, 1, Z), 128, (size_t)M * (M / 2) * sizeof(float), s>>>(
        a.src, llin, ll, a.U, n, M, j == 0, last, kk, rho);
  }
}

cudaError_t launch_dwt_analysis(const Geom& g, const DwtArgs& a, int mode, cudaStream_t s) {
  for (int j = 0; j < g.J; ++j) {
    if (mode == MODE_UPDATE) dwt_level<MODE_UPDATE>(g, a, j, s);
    else dwt_level<MODE_LINEAR>(g, a, j, s);
  }
  return cudaGetLastError();
}

cudaError_t launch_dwt_adjoint(const Geom& g, const DwtArgs& a, cudaStream_t s) {
  const int n = g.n, Z = kDbBases * g.L;
  const float* in = a.W2;       // low-low images of the level before
  for (int j = g.J - 1; j >= 0; --j) {
    const int M = n >> j, coarsest = j == g.J - 1;
    if (M >= kMinTile) {
      float* out = j == 0 ? a.S : in == a.W1 ? a.W2 : a.W1;
      // rows per group: 16, as many threads as columns; 8 at 1024 columns (512 threads, two columns each)
      const size_t sm = (size_t)syn_pitch(M) * sizeof(float);
      if (j > 0) k_idwt_group<16><<<dim3(M / 16, 1, Z), M, 16 * sm, s>>>(a.U, in, out, n, M, coarsest);
      else if (M == 1024) k_idwt_group_sum<8><<<dim3(M / 8, 1, g.L), 512, 8 * sm, s>>>(a.U, in, out, n, coarsest);
      else k_idwt_group_sum<16><<<dim3(M / 16, 1, g.L), M, 16 * sm, s>>>(a.U, in, out, n, coarsest);
      in = out;
      continue;
    }
    // small levels come first and hand their images on in W2
    k_idwt_cols<<<dim3(1, 1, Z), dim3(32, 8), 0, s>>>(a.U, a.W2, a.W1, n, M, coarsest);
    if (j > 0) k_idwt_rows<<<dim3(1, (M + kRowsPerBlock - 1) / kRowsPerBlock, Z), 64, 0, s>>>(a.W1, a.W2, n, M);
    else k_idwt_rows_sum<<<dim3(1, (M + kRowsPerBlock - 1) / kRowsPerBlock, g.L), 64, 0, s>>>(a.W1, a.S, n);
  }
  return cudaGetLastError();
}

// Kernels that one analysis and one adjoint launch.
int dwt_kernels(const Geom& g) {
  int k = g.J;
  for (int j = 0; j < g.J; ++j) k += (g.n >> j) >= kMinTile ? 1 : 2;
  return k;
}

cudaError_t launch_abs_sum(const float* x, size_t n, double* partials, int* nparts, cudaStream_t s) {
  const int blocks = (int)std::min<size_t>((n + 255) / 256, 1024);
  k_abs_sum<<<blocks, 256, 0, s>>>(x, n, partials);
  if (nparts) *nparts = blocks;
  return cudaGetLastError();
}

}  // namespace muffin

extern "C" int muffin_daubechies_filter(int p, double* h_out) {
  return muffin::daubechies_lowpass(p, h_out) ? 0 : -1;
}
