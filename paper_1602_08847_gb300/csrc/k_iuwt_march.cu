// Fine levels of the generation-1 IUWT (Eqs. 9 and 11) as a march down the
// rows of whole-width strips, for images of at least 128 columns.
//
// A block owns rows y0 .. y1-1 of one channel over the full width N: thread t
// holds columns 4t .. 4t+3 and walks down the rows, one row per step.  Every
// level j keeps the last 4D rows (D = 2^j) of its input, private to the
// thread: in registers up to 4D = 8, in shared memory above.  One step
//   1. forms the vertical five-tap sum of every level from its ring and the
//      row that has just come in, and writes it to shared memory;
//   2. one barrier;
//   3. forms the horizontal sum from the neighbours' chunks (full width, so
//      the periodic wrap is a mask on the chunk index), and from it the next
//      level's input row, which that level takes up in the next step.
// The levels run skewed by one step, so one barrier per row serves them all
// (the vertical sums are double buffered).  Against 64 x 64 halo tiles there
// is no horizontal halo, the vertical one is paid once per strip instead of
// once per tile (2H rows; the tiles filter 2.1 times their area), a row costs
// one barrier instead of six, and every global access is a whole row.
// Sums are taken in the order of the tile kernels (iuwt_vec.cuh): the results
// are bitwise theirs.
//
// Measured at 512 x 512 x 256, three fine levels (us per launch, tiles before,
// march now, bytes each must move): analysis 490 -> 362 (2.15 GB: 5.9 TB/s, DRAM
// bound), adjoint 670 -> 286 (1.34 GB: 4.7 TB/s; 12 warps per SM, bound by the
// latency and the issue slots of a step; three levels spill 36 bytes a thread at
// 168 registers for N below 1024).  256 x 256 x 64, two levels: 28.7 ->
// 22.8 and 40.9 -> 21.0.

#include "internal.h"
#include "iuwt_vec.cuh"

namespace muffin {
namespace march {

using vec::b3u;
using vec::b3u4;
using vec::dual4;
using vec::ld4;
using vec::ldg4;
using vec::st4;
using vec::sub4;

constexpr int kUnroll = 8;     // steps per trip of the row loop: ring slots up to 8 rows are fixed at compile time
// Rows between a row's L2 prefetch and its use: long enough for DRAM under load,
// short enough to be still there.  512x512x256, three levels, ms per launch:
// analysis 0.362 / 0.380 / 0.384 / 0.392 / 0.421 / 0.479 and adjoint 0.302 /
// 0.286 / 0.288 / 0.288 / 0.303 / 0.397 at 2 / 3 / 4 / 6 / 8 / 14 rows.
constexpr int kAheadAn = 2, kAheadAdj = 3;

template <int N, int J1> struct Strip {
  static constexpr int NT = N / 4;
  static constexpr int H = (2 << J1) - 2;              // rows of halo above and below the strip
  static constexpr int LAG = 2 * H + J1 - 1;           // steps before and after the strip's own rows
  static constexpr int RING = J1 == 3 ? 16 : 0;        // rows of shared ring (level 2 only)
  static constexpr size_t SMEM = (size_t)(RING + 2 * J1) * N * sizeof(float);
  // the adjoint also keeps the u_j rows between their first use and their second, 2D rows later
  static constexpr int DELAY = (2 << J1) - 2;
  static constexpr size_t SMEM_ADJ = SMEM + (size_t)DELAY * N * sizeof(float);
  // blocks per SM: 16 warps of 128 registers (analysis), 12 warps (adjoint, by shared memory)
  static constexpr int MINB = 2048 / N;
  static constexpr int MINB_ADJ = N == 1024 ? 1 : 1536 / N;
};

// Vertical ring of one level: the last 4D input rows.
template <int D> struct RegRing {
  float4 v[4 * D];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int i = 0; i < 4 * D; ++i) v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // takes row x of step K (mod the unroll); returns the vertical sum, mid: the row 2D back
  template <int K> __device__ __forceinline__ float4 push(float4 x, float4* mid) {
    constexpr int S = K % (4 * D);
    const float4 c = v[(S + 2 * D) % (4 * D)];
    const float4 r = b3u4(v[S], v[(S + D) % (4 * D)], c, v[(S + 3 * D) % (4 * D)], x);
    v[S] = x;
    *mid = c;
    return r;
  }
};

// Level 2 (D = 4): 16 rows of pitch N; lo / hi: the half the current trip's
// eight steps write, and the other one (they swap every trip).
template <int N, int K>
__device__ __forceinline__ float4 push_shared(float* lo, float* hi, float4 x, float4* mid) {
  constexpr int D = 4;
  auto row = [&](int i) { return i < 8 ? lo + i * N : hi + (i - 8) * N; };
  float* p = row(K);
  const float4 a = ld4(p), b = ld4(row((K + D) & 15)), c = ld4(row((K + 2 * D) & 15)), d = ld4(row((K + 3 * D) & 15));
  st4(p, x);
  *mid = c;
  return b3u4(a, b, c, d, x);
}

// Horizontal sum of chunk t of a row of vertical sums (own: this thread's chunk).
template <int N, int D> __device__ __forceinline__ float4 hrow(const float* row, float4 own, int t) {
  constexpr int M = N / 4 - 1;
  if constexpr (D == 1) {
    const float2 l = *reinterpret_cast<const float2*>(row + 4 * ((t - 1) & M) + 2);
    const float2 r = *reinterpret_cast<const float2*>(row + 4 * ((t + 1) & M));
    return make_float4(b3u(l.x, l.y, own.x, own.y, own.z), b3u(l.y, own.x, own.y, own.z, own.w),
                       b3u(own.x, own.y, own.z, own.w, r.x), b3u(own.y, own.z, own.w, r.x, r.y));
  } else if constexpr (D == 2) {
    const float4 l = ld4(row + 4 * ((t - 1) & M)), r = ld4(row + 4 * ((t + 1) & M));
    return make_float4(b3u(l.x, l.z, own.x, own.z, r.x), b3u(l.y, l.w, own.y, own.w, r.y),
                       b3u(l.z, own.x, own.z, r.x, r.z), b3u(l.w, own.y, own.w, r.y, r.w));
  } else {
    const float4 l2 = ld4(row + 4 * ((t - 2) & M)), l = ld4(row + 4 * ((t - 1) & M));
    const float4 r = ld4(row + 4 * ((t + 1) & M)), r2 = ld4(row + 4 * ((t + 2) & M));
    return b3u4(l2, l, own, r, r2);
  }
}

__device__ __forceinline__ float4 scale256(float4 v) {
  constexpr float inv = 1.0f / 256.0f;
  return make_float4(v.x * inv, v.y * inv, v.z * inv, v.w * inv);
}

// Address of pixel (gy, 4t + i) of a class-permuted plane (stride 2^J1).
template <int N, int J1> __device__ __forceinline__ size_t class_at(int gy, int t, int i) {
  constexpr int S = 1 << J1, mc = N >> J1;
  const int x = 4 * t + i;
  return (size_t)((gy & (S - 1)) * S + (x & (S - 1))) * mc * mc + (size_t)(gy >> J1) * mc + (x >> J1);
}

// ------------------------------------------------------------------ analysis and spatial dual update
// LAST: the coarse plane is c_J1 itself (J == J1), its dual U_J is updated here.
template <int N, int J1, bool LAST> struct Analysis {
  using G = Strip<N, J1>;
  // rows between level 0's input and level j's output
  __host__ __device__ static constexpr int OFF(int j) { return (4 << j) - 2 + j; }
  const float* D;
  float* U;          // U_0 of the channel, at column 4t
  float* cls;        // class-permuted plane that c_J1 (or U_J) goes to
  float* ring;       // shared ring of level 2, at column 4t
  float* tb;         // vertical sums [2][J1][N]
  int t, y0, y1;
  float k, rho;

  RegRing<1> r0;
  RegRing<2> r1;
  float4 x[J1], u[J1];
  float uc[LAST ? 4 : 1];      // U_J beside u[J1 - 1]

  // the rows before the first ones that the steps prefetch, into L2 at once
  __device__ __forceinline__ void ahead() const {
    if ((t & 7) != 0) return;
    for (int i = 1; i < kAheadAn; ++i) pf_line(D + (size_t)((y0 - G::H + i) & (N - 1)) * N);
  }

  template <int K> __device__ __forceinline__ void step(int s, float* lo, float* hi) {
    const int e0 = y0 - G::H + s;
    // next step's rows
    const float4 xn = ldg4(D + (size_t)((e0 + 1) & (N - 1)) * N);
    float4 un[J1];
#pragma unroll
    for (int j = 0; j < J1; ++j) {
      const int o = e0 + 1 - OFF(j);
      un[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (o >= y0 && o < y1) un[j] = ldg4(U + (size_t)j * N * N + (size_t)o * N);
    }
    float ucn[LAST ? 4 : 1] = {};
    if constexpr (LAST) {
      const int o = e0 + 1 - OFF(J1 - 1);
      if (o >= y0 && o < y1)
#pragma unroll
        for (int i = 0; i < 4; ++i) ucn[i] = __ldcg(cls + class_at<N, J1>(o, t, i));
    }
    if ((t & 7) == 0) {
      pf_line(D + (size_t)((e0 + kAheadAn) & (N - 1)) * N);
#pragma unroll
      for (int j = 0; j < J1; ++j) {
        const int o = e0 + kAheadAn - OFF(j);
        if (o >= y0 && o < y1) pf_line(U + (size_t)j * N * N + (size_t)o * N);
      }
    }
    float4 mid[J1], own[J1];
    own[0] = r0.template push<K>(x[0], &mid[0]);
    if constexpr (J1 > 1) own[1] = r1.template push<K>(x[1], &mid[1]);
    if constexpr (J1 > 2) own[2] = push_shared<N, K>(lo, hi, x[2], &mid[2]);
    float* tw = tb + (K & 1) * J1 * N;
#pragma unroll
    for (int j = 0; j < J1; ++j) st4(tw + j * N + 4 * t, own[j]);
    __syncthreads();
#pragma unroll
    for (int j = 0; j < J1; ++j) {
      float4 raw;
      if (j == 0) raw = hrow<N, 1>(tw, own[0], t);
      else if (j == 1) raw = hrow<N, 2>(tw + N, own[j], t);
      else raw = hrow<N, 4>(tw + 2 * N, own[j], t);
      const float4 cn = scale256(raw);
      const int o = e0 - OFF(j);
      if (o >= y0 && o < y1) {
        st4(U + (size_t)j * N * N + (size_t)o * N, dual4(u[j], sub4(mid[j], cn), k, rho));
        if (j == J1 - 1) {
          float v[4] = {cn.x, cn.y, cn.z, cn.w};
#pragma unroll
          for (int i = 0; i < 4; ++i)
            cls[class_at<N, J1>(o, t, i)] = LAST ? vec::dual1(uc[LAST ? i : 0], v[i], k, rho) : v[i];
        }
      }
      if (j + 1 < J1) x[j + 1] = cn;
    }
    x[0] = xn;
#pragma unroll
    for (int j = 0; j < J1; ++j) u[j] = un[j];
    if constexpr (LAST)
#pragma unroll
      for (int i = 0; i < 4; ++i) uc[i] = ucn[i];
  }
};

// grid (strips, L); U: [L][J+1][N][N], planes j >= J1 class-permuted
template <int N, int J1, bool LAST>
__global__ void __launch_bounds__(N / 4, Strip<N, J1>::MINB)
k_fine_analysis_m(int J, const float* __restrict__ D, float* __restrict__ U, float* __restrict__ cr, float k, float rho,
                  int rows) {
  using G = Strip<N, J1>;
  extern __shared__ __align__(16) float sm[];
  constexpr size_t P = (size_t)N * N;
  const int l = blockIdx.y;
  Analysis<N, J1, LAST> a;
  a.t = threadIdx.x;
  a.y0 = blockIdx.x * rows;
  a.y1 = min(N, a.y0 + rows);
  a.D = D + (size_t)l * P + 4 * a.t;
  a.U = U + (size_t)l * (J + 1) * P + 4 * a.t;
  a.cls = LAST ? U + ((size_t)l * (J + 1) + J) * P : cr + (size_t)l * P;
  a.tb = sm;
  a.ring = sm + 2 * J1 * N + 4 * a.t;
  a.k = k;
  a.rho = rho;
  a.ahead();
  a.r0.clear();
  a.r1.clear();
#pragma unroll
  for (int j = 0; j < J1; ++j) a.x[j] = a.u[j] = make_float4(0.f, 0.f, 0.f, 0.f);
  a.x[0] = ldg4(a.D + (size_t)((a.y0 - G::H) & (N - 1)) * N);
  for (float& v : a.uc) v = 0.f;
#pragma unroll
  for (int i = 0; i < G::RING; ++i) st4(a.ring + i * N, make_float4(0.f, 0.f, 0.f, 0.f));
  float *lo = a.ring, *hi = a.ring + 8 * N;
  const int steps = a.y1 - a.y0 + G::LAG;
  for (int s = 0; s < steps; s += kUnroll) {
    a.template step<0>(s, lo, hi);
    a.template step<1>(s + 1, lo, hi);
    a.template step<2>(s + 2, lo, hi);
    a.template step<3>(s + 3, lo, hi);
    a.template step<4>(s + 4, lo, hi);
    a.template step<5>(s + 5, lo, hi);
    a.template step<6>(s + 6, lo, hi);
    a.template step<7>(s + 7, lo, hi);
    float* w = lo;
    lo = hi;
    hi = w;
  }
}

// ------------------------------------------------------------------ adjoint
// r_j = u_j + H_j (r_{j+1} - u_j) for j = J1-1 .. 0, from r_J1 (class-permuted); S = r_0.
template <int N, int J1> struct Adjoint {
  using G = Strip<N, J1>;
  // rows between the r_J1 row of a step and level j's output / input row
  __host__ __device__ static constexpr int OFF(int j) { return (4 << (J1 - 1)) - (2 << j) + J1 - 1 - j; }
  __host__ __device__ static constexpr int IN(int j) { return j == J1 - 1 ? 0 : OFF(j + 1) + 1; }
  const float* rin;  // class-permuted plane of the channel
  const float* U;    // U_0 of the channel, at column 4t
  float* S;          // at column 4t
  float* ring;
  float* tb;
  int t, y0, y1;

  RegRing<1> r0;
  RegRing<2> r1;
  float* delay;      // u_j rows of the last 2D steps, levels one after another, at column 4t
  float4 q[J1];      // the r_{j+1} - u_j row that level j takes up in this step
  float4 uc[J1];     // u_j at the row that level j completes in this step

  // the rows before the first ones that the steps prefetch, into L2 at once
  __device__ __forceinline__ void ahead() const {
    if ((t & 7) != 0) return;
    for (int i = 0; i < kAheadAdj; ++i) {
      pf_line(U + (size_t)(J1 - 1) * N * N + (size_t)((y0 - G::H + i) & (N - 1)) * N);
      pf_r(y0 - G::H + i);
    }
  }
  __device__ __forceinline__ void pf_r(int e) const {
    constexpr int SC = 1 << J1, mc = N >> J1;
    const int gy = e & (N - 1), i = t >> 3, c = i % SC, part = i / SC;
    pf_line(rin + (size_t)((gy & (SC - 1)) * SC + c) * mc * mc + (size_t)(gy >> J1) * mc + 32 * part);
  }
  __device__ __forceinline__ float4 load_r(int e) const {
    const int gy = e & (N - 1);
    return make_float4(__ldcg(rin + class_at<N, J1>(gy, t, 0)), __ldcg(rin + class_at<N, J1>(gy, t, 1)),
                       __ldcg(rin + class_at<N, J1>(gy, t, 2)), __ldcg(rin + class_at<N, J1>(gy, t, 3)));
  }
  __device__ __forceinline__ float4 load_u(int j, int row) const {
    return ldg4(U + (size_t)j * N * N + (size_t)(row & (N - 1)) * N);
  }

  template <int K> __device__ __forceinline__ void step(int s, float* lo, float* hi) {
    const int e = y0 - G::H + s;
    // next step's rows
    const float4 rn = load_r(e + 1);
    float4 un[J1];
#pragma unroll
    for (int j = 0; j < J1; ++j) un[j] = load_u(j, e + 1 - IN(j));
    if ((t & 7) == 0) {
#pragma unroll
      for (int j = 0; j < J1; ++j) pf_line(U + (size_t)j * N * N + (size_t)((e + kAheadAdj - IN(j)) & (N - 1)) * N);
      pf_r(e + kAheadAdj);
    }
    float4 own[J1], mid;
    own[0] = r0.template push<K>(q[0], &mid);
    if constexpr (J1 > 1) own[1] = r1.template push<K>(q[1], &mid);
    if constexpr (J1 > 2) own[2] = push_shared<N, K>(lo, hi, q[2], &mid);
    float* tw = tb + (K & 1) * J1 * N;
#pragma unroll
    for (int j = 0; j < J1; ++j) st4(tw + j * N + 4 * t, own[j]);
    __syncthreads();
    constexpr float inv = 1.0f / 256.0f;
#pragma unroll
    for (int j = 0; j < J1; ++j) {
      float4 raw;
      if (j == 0) raw = hrow<N, 1>(tw, own[0], t);
      else if (j == 1) raw = hrow<N, 2>(tw + N, own[j], t);
      else raw = hrow<N, 4>(tw + 2 * N, own[j], t);
      const float4 v = make_float4(fmaf(raw.x, inv, uc[j].x), fmaf(raw.y, inv, uc[j].y), fmaf(raw.z, inv, uc[j].z),
                                   fmaf(raw.w, inv, uc[j].w));
      if (j > 0) q[j - 1] = sub4(v, un[j - 1]);
      else {
        const int o = e - OFF(0);
        if (o >= y0 && o < y1) st4(S + (size_t)o * N, v);
      }
    }
    q[J1 - 1] = sub4(rn, un[J1 - 1]);
    // the row of the next step into the delay line, the row 2D before it out
#pragma unroll
    for (int j = 0; j < J1; ++j) {
      float* p = delay + ((2 << j) - 2 + ((K + 1) & ((2 << j) - 1))) * N;
      uc[j] = ld4(p);
      st4(p, un[j]);
    }
  }
};

// strips > 0: block b takes strip b % strips of channel b / strips; strips = 0:
// rows b * rows .. of the channels taken one after another (L * N rows in all),
// starting over at a channel's end.
template <int N, int J1>
__global__ void __launch_bounds__(N / 4, Strip<N, J1>::MINB_ADJ)
k_fine_adjoint_m(int J, int L, const float* __restrict__ rin, size_t rin_stride, const float* __restrict__ U,
                 float* __restrict__ S, int rows, int strips) {
  using G = Strip<N, J1>;
  extern __shared__ __align__(16) float sm[];
  constexpr size_t P = (size_t)N * N;
  Adjoint<N, J1> a;
  a.t = threadIdx.x;
  a.tb = sm;
  a.ring = sm + 2 * J1 * N + 4 * a.t;
  a.delay = a.ring + G::RING * N;
  a.r0.clear();
  a.r1.clear();
#pragma unroll
  for (int j = 0; j < J1; ++j) a.q[j] = a.uc[j] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < G::RING + G::DELAY; ++i) st4(a.ring + i * N, make_float4(0.f, 0.f, 0.f, 0.f));
  float *lo = a.ring, *hi = a.ring + 8 * N;
  int row, end;
  if (strips > 0) {
    const int l = blockIdx.x / strips;
    row = l * N + (blockIdx.x % strips) * rows;
    end = min((l + 1) * N, row + rows);
  } else {
    row = blockIdx.x * rows;
    end = min(L * N, row + rows);
  }
  while (row < end) {
    const int l = row / N;
    a.y0 = row % N;
    a.y1 = min(N, a.y0 + end - row);
    row += a.y1 - a.y0;
    a.rin = rin + (size_t)l * rin_stride;
    a.U = U + (size_t)l * (J + 1) * P + 4 * a.t;
    a.S = S + (size_t)l * P + 4 * a.t;
    a.ahead();
    const float4 u0 = a.load_u(J1 - 1, a.y0 - G::H);
    a.q[J1 - 1] = sub4(a.load_r(a.y0 - G::H), u0);
    st4(a.delay + ((1 << J1) - 2) * N, u0);      // slot 0 of the level's delay line
    const int steps = a.y1 - a.y0 + G::LAG;
    for (int s = 0; s < steps; s += kUnroll) {
      a.template step<0>(s, lo, hi);
      a.template step<1>(s + 1, lo, hi);
      a.template step<2>(s + 2, lo, hi);
      a.template step<3>(s + 3, lo, hi);
      a.template step<4>(s + 4, lo, hi);
      a.template step<5>(s + 5, lo, hi);
      a.template step<6>(s + 6, lo, hi);
      a.template step<7>(s + 7, lo, hi);
      float* w = lo;
      lo = hi;
      hi = w;
    }
  }
}

}  // namespace march

// ------------------------------------------------------------------ host side
// How a kernel's rows are split over blocks.  A step (one row of every
// resident block) was measured to take about lat + warp * (warps on the SM)
// microseconds; the cheapest in steps times step time wins.
struct Split { int rows, strips; };
struct StepTime { float lat, warp; };
// by the number of levels (strip counts of 1 to 32 timed on 512 x 512 x {4, 8, 64, 256},
// 256 x 256 x {16, 32, 64}, 1024 x 1024 x {2, 8, 64}, 128 x 128 x {64, 128})
constexpr StepTime kAnalysisStep[4] = {{}, {0.30f, 0.020f}, {0.38f, 0.024f}, {0.50f, 0.045f}};
constexpr StepTime kAdjointStep[4] = {{}, {0.30f, 0.020f}, {0.33f, 0.030f}, {0.27f, 0.050f}};

static Split split_rows(int n, int L, int lag, int minb, StepTime t, bool chunks) {
  const int sms = device_sms();
  auto steps = [&](int rows) { return (rows + lag + march::kUnroll - 1) / march::kUnroll * march::kUnroll + 2; };
  Split best{n, 1};
  float best_cost = 1e30f;
  for (int strips = 1; strips <= 32 && strips * 4 <= n; ++strips) {
    const int rows = (n + strips - 1) / strips, on = (L * strips + sms - 1) / sms, k = on < minb ? on : minb;
    const float cost = (float)((on + minb - 1) / minb) * steps(rows) * (t.lat + t.warp * k * (n / 128));
    if (cost < best_cost) { best_cost = cost; best = Split{rows, strips}; }
  }
  if (chunks) {
    // every block the same number of rows, most of them over a channel's end
    const int rows = (L * n + sms * minb - 1) / (sms * minb);
    if (rows >= 8 && (steps(rows) + steps(0)) * (t.lat + t.warp * minb * (n / 128)) < best_cost) best = Split{rows, 0};
  }
  return best;
}

// Where the march is taken.  A strip costs its LAG rows and a step some 0.3 us
// whatever its occupancy, so small cubes stay on the halo tiles.  Both sides
// measured (us per launch, tiles / march): adjoint 256x256x16 12.5 / 14.5,
// 256x256x32 20.7 / 16.5, 128x128x128 14.2 / 10.4, 512x512x8 30.8 / 28.9;
// analysis 256x256x32 16.6 / 16.8, 256x256x64 28.7 / 22.8, 512x512x8 24.5 / 33,
// 1024x1024x8 73.7 / 69.8.
static bool march_fits(const Geom& g) { return g.vec && g.gen == 1 && g.n >= 128 && g.j1 >= 1 && g.j1 <= 3 && g.J >= g.j1; }
bool iuwt_march_analysis(const Geom& g) { return march_fits(g) && (size_t)g.L * g.n * g.n >= ((size_t)1 << 22); }
bool iuwt_march_adjoint(const Geom& g) { return march_fits(g) && (size_t)g.L * g.n * g.n >= ((size_t)1 << 21); }

#define MARCH_CASES(F)                                              \
  switch (g.n * 4 + g.j1) {                                         \
    case 128 * 4 + 1: F(128, 1) case 128 * 4 + 2: F(128, 2) case 128 * 4 + 3: F(128, 3)    \
    case 256 * 4 + 1: F(256, 1) case 256 * 4 + 2: F(256, 2) case 256 * 4 + 3: F(256, 3)    \
    case 512 * 4 + 1: F(512, 1) case 512 * 4 + 2: F(512, 2) case 512 * 4 + 3: F(512, 3)    \
    case 1024 * 4 + 1: F(1024, 1) case 1024 * 4 + 2: F(1024, 2) case 1024 * 4 + 3: F(1024, 3) \
  }                                                                 \
  return cudaErrorInvalidValue;

cudaError_t launch_fine_analysis_march(const Geom& g, const IuwtArgs& a, cudaStream_t s) {
#define FA(NN, JJ)                                                                                       \
  {                                                                                                      \
    using G = march::Strip<NN, JJ>;                                                                      \
    const Split p = split_rows(NN, g.L, G::LAG, G::MINB, kAnalysisStep[JJ], false);                      \
    const dim3 grid(p.strips, g.L);                                                                      \
    if (g.J == JJ)                                                                                       \
      march::k_fine_analysis_m<NN, JJ, true><<<grid, NN / 4, G::SMEM, s>>>(g.J, a.D, a.U, a.cr, a.k, a.rho, p.rows); \
    else                                                                                                 \
      march::k_fine_analysis_m<NN, JJ, false><<<grid, NN / 4, G::SMEM, s>>>(g.J, a.D, a.U, a.cr, a.k, a.rho, p.rows); \
    return cudaGetLastError();                                                                           \
  }
  MARCH_CASES(FA)
#undef FA
}

cudaError_t launch_fine_adjoint_march(const Geom& g, const IuwtArgs& a, cudaStream_t s) {
  const size_t P = (size_t)g.n * g.n;
  const bool from_u = g.J == g.j1;
  const float* rin = from_u ? a.U + (size_t)g.J * P : a.rin;
  const size_t stride = from_u ? (size_t)(g.J + 1) * P : P;
#define FT(NN, JJ)                                                                                       \
  {                                                                                                      \
    using G = march::Strip<NN, JJ>;                                                                      \
    const Split p = split_rows(NN, g.L, G::LAG, G::MINB_ADJ, kAdjointStep[JJ], true);                                      \
    const int blocks = p.strips > 0 ? g.L * p.strips : (g.L * NN + p.rows - 1) / p.rows;                 \
    march::k_fine_adjoint_m<NN, JJ><<<blocks, NN / 4, G::SMEM_ADJ, s>>>(g.J, g.L, rin, stride, a.U, a.S, p.rows, \
                                                                        p.strips);                       \
    return cudaGetLastError();                                                                           \
  }
  MARCH_CASES(FT)
#undef FT
}

cudaError_t iuwt_march_configure(const Geom& g) {
  if (!march_fits(g)) return cudaSuccess;
#define SET(NN, JJ)                                                                       \
  {                                                                                       \
    cudaError_t e = allow_max_dyn_smem(march::k_fine_analysis_m<NN, JJ, true>);           \
    if (e == cudaSuccess) e = allow_max_dyn_smem(march::k_fine_analysis_m<NN, JJ, false>); \
    return e != cudaSuccess ? e : allow_max_dyn_smem(march::k_fine_adjoint_m<NN, JJ>);    \
  }
  MARCH_CASES(SET)
#undef SET
}

}  // namespace muffin
