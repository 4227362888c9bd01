// Coarse levels of the generation-1 IUWT on 128 x 128 class sub-images as a
// march of single warps: analysis with the dual updates, and the adjoint of the
// updated duals right behind it.
//
// A row of a sub-image is 32 chunks of four columns, one per lane; a warp walks
// down the rows, one a step.  Every level keeps the last 4d rows of its input
// (d = 2^level) private to the lane, level 0 in registers, level 1 in shared
// memory; the horizontal neighbours come by shuffles, whose lane index wraps as
// the periodic row does.  Nothing is shared between lanes through memory, so
// there is no barrier, and 12 to 20 warps an SM work on as many sub-images
// where a block per sub-image that holds it whole (k_coarse_s: 137 KB) leaves
// 16 warps waiting at one block's barriers.  Levels and adjoint levels run
// skewed by one step.
//
// Rows are counted on past M: the analysis covers rows 0 .. M-1 (reading A =
// 2 (2^NL - 1) rows of halo before and after), the adjoint rows A .. M+A-1,
// whose inputs it takes from the analysis as they appear, and past row M-1 from
// the dual planes written at the start.  A row of r_out is written after the
// last read of that row of c_in (they may be one array).  Sums are taken in the
// order of the block kernels (iuwt_vec.cuh): the results are bitwise theirs.
//
// Measured (block kernel, march; one level moves 24 bytes a voxel, two 32):
// 1024 x 1024 x 64, two levels 1085 -> 433 us (5.0 TB/s), 1024 x 1024 x 8, one
// level 96.7 -> 64.9 us (512 warps: bound by the latency of a step).  A warp's
// rows are a serial chain, so few sub-images stay with the block kernel
// (1024 x 1024 x 4, two levels: 80.2 against 84.6 us; x 2, one level: 28.0
// against 61.0).  The same march on 64 x 64 sub-images, two to a warp, was no
// faster than their resident kernel (512 x 512 x 256, two levels: 454 against
// 457 us), with three levels it spills and loses everywhere.
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

constexpr int kCoarseWarps = 4;     // warps of a block (independent of one another)
// Rows between a row's L2 prefetch and its use.  1024x1024x64, two levels / one
// level, us per launch in a pass: 587 / 415 at 1 row, 493 / 378 at 2, 485 / 374 at
// 3, 487 / 375 at 4, 491 / 390 at 6, 509 / 386 at 8.
constexpr int kAheadCoarse = 4;
constexpr int M = 128;              // side of a sub-image

template <int NL> struct CoarseM {
  __host__ __device__ static constexpr int A() { return 2 * ((1 << NL) - 1); }
  // rows between the input row of a step and level j's output, the adjoint's input and its output
  __host__ __device__ static constexpr int OFF(int j) { return (4 << j) - 2 + j; }
  __host__ __device__ static constexpr int OA(int j) {
    return j == NL - 1 ? OFF(NL - 1) + 1 + (2 << j) : OA(j + 1) + 1 + (2 << j);
  }
  __host__ __device__ static constexpr int IA(int j) { return j == NL - 1 ? OFF(NL - 1) + 1 : OA(j + 1) + 1; }
  // shared rings of level 1, 8 rows each, analysis and adjoint
  static constexpr int ROWS = NL == 1 ? 0 : 16;
  static constexpr size_t SMEM = (size_t)kCoarseWarps * ROWS * M * sizeof(float);
};

__device__ __forceinline__ float4 shfl4(float4 v, int lane) {
  return make_float4(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane),
                     __shfl_sync(0xffffffffu, v.z, lane), __shfl_sync(0xffffffffu, v.w, lane));
}

// Horizontal sum at dilation 1 << LV.
template <int LV> __device__ __forceinline__ float4 hsum_warp(float4 v, int lane) {
  const int l = (lane - 1) & 31, r = (lane + 1) & 31;
  if constexpr (LV == 0) {
    const float lz = __shfl_sync(0xffffffffu, v.z, l), lw = __shfl_sync(0xffffffffu, v.w, l);
    const float rx = __shfl_sync(0xffffffffu, v.x, r), ry = __shfl_sync(0xffffffffu, v.y, r);
    return make_float4(b3u(lz, lw, v.x, v.y, v.z), b3u(lw, v.x, v.y, v.z, v.w), b3u(v.x, v.y, v.z, v.w, rx),
                       b3u(v.y, v.z, v.w, rx, ry));
  } else {
    const float4 p = shfl4(v, l), q = shfl4(v, r);
    return make_float4(b3u(p.x, p.z, v.x, v.z, q.x), b3u(p.y, p.w, v.y, v.w, q.y), b3u(p.z, v.x, v.z, q.x, q.z),
                       b3u(p.w, v.y, v.w, q.y, q.w));
  }
}

// Vertical sum of level LV with row x of step s; mid: the row 2d back.  reg:
// level 0's ring (slot K), sm: the shared ring of level 1 (4d rows of 128 floats).
template <int LV, int K>
__device__ __forceinline__ float4 vsum(float4 (&reg)[4], float* sm, int s, float4 x, float4* mid) {
  if constexpr (LV == 0) {
    const float4 c = reg[(K + 2) & 3];
    const float4 r = b3u4(reg[K], reg[(K + 1) & 3], c, reg[(K + 3) & 3], x);
    reg[K] = x;
    *mid = c;
    return r;
  } else {
    constexpr int d = 1 << LV, mask = 4 * d - 1;
    float* p = sm + (s & mask) * M;
    const float4 a = ld4(p), b = ld4(sm + ((s + d) & mask) * M), c = ld4(sm + ((s + 2 * d) & mask) * M),
                 e = ld4(sm + ((s + 3 * d) & mask) * M);
    st4(p, x);
    *mid = c;
    return b3u4(a, b, c, e, x);
  }
}

template <int NL> struct CoarseWarp {
  using G = CoarseM<NL>;
  const float* cin;    // the lane's chunk of row 0
  float* rout;
  float* U;            // U_j1 of the sub-image, same chunk
  size_t plane;
  float* ring;         // shared rings, at this lane's chunk
  int lane;
  float k, rho;
  float4 ra[4], rb[4];           // level 0's rings, analysis and adjoint
  float4 x[NL], u[NL + 1];       // rows the analysis levels take up; old duals of their output rows (u[NL]: U_J)
  float4 q[NL];                  // r_{j+1} - u_j rows the adjoint levels take up
  float4 ui[NL], uc[NL];         // u_j at the row r_{j+1} - u_j is next formed for (j < NL - 1); at the row completed

  __device__ __forceinline__ float4 dual_row(int j, int row) const {
    return ldg4(U + (size_t)j * plane + (size_t)(row & (M - 1)) * M);
  }

  template <int LV, int K> __device__ __forceinline__ void analysis(int s, int e, float4* cn_out, float4* un_out) {
    float4 mid;
    const float4 v = vsum<LV, K>(ra, ring, s, x[LV], &mid);
    const float4 raw = hsum_warp<LV>(v, lane);
    constexpr float inv = 1.0f / 256.0f;
    const float4 cn = make_float4(raw.x * inv, raw.y * inv, raw.z * inv, raw.w * inv);
    const int o = e - G::OFF(LV);
    *un_out = dual4(u[LV], sub4(mid, cn), k, rho);
    if (o >= 0 && o < M) st4(U + (size_t)LV * plane + (size_t)o * M, *un_out);
    *cn_out = cn;
  }

  template <int LV, int K> __device__ __forceinline__ float4 adjoint(int s) {
    float4 mid;
    const float4 v = vsum<LV, K>(rb, ring + 8 * M, s, q[LV], &mid);
    const float4 raw = hsum_warp<LV>(v, lane);
    constexpr float inv = 1.0f / 256.0f;
    return make_float4(fmaf(raw.x, inv, uc[LV].x), fmaf(raw.y, inv, uc[LV].y), fmaf(raw.z, inv, uc[LV].z),
                       fmaf(raw.w, inv, uc[LV].w));
  }

  template <int K> __device__ __forceinline__ void step(int s) {
    const int e = s - G::A();
    // next step's rows: c, the old duals, and the new duals that the adjoint reads back (written long before)
    float4 xn = make_float4(0.f, 0.f, 0.f, 0.f), un[NL + 1], uin[NL], ucn[NL];
    if (e + 1 < M + G::A()) xn = ldg4(cin + (size_t)((e + 1) & (M - 1)) * M);
#pragma unroll
    for (int j = 0; j <= NL; ++j) {
      const int o = e + 1 - G::OFF(j < NL ? j : NL - 1);
      un[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (o >= 0 && o < M) un[j] = ldg4(U + (size_t)j * plane + (size_t)o * M);
      // past the last row: the planes' new values, for the adjoint's topmost input
      else if (j >= NL - 1 && o >= M) un[j] = dual_row(j, o);
    }
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      uin[j] = ucn[j] = make_float4(0.f, 0.f, 0.f, 0.f);
      const int oc = e + 1 - G::OA(j), oi = e + 2 - G::IA(j);
      if (oc >= 0) ucn[j] = dual_row(j, oc);
      if (j < NL - 1 && oi >= 0) uin[j] = dual_row(j, oi);
    }
    // and, some rows ahead, what comes from DRAM into L2
    if ((lane & 7) == 0) {
      if (e + kAheadCoarse < M) pf_line(cin + (size_t)((e + kAheadCoarse) & (M - 1)) * M);
#pragma unroll
      for (int j = 0; j <= NL; ++j) {
        const int o = e + kAheadCoarse - G::OFF(j < NL ? j : NL - 1);
        if (o >= 0 && o < M) pf_line(U + (size_t)j * plane + (size_t)o * M);
      }
    }
    // adjoint levels, then analysis levels (each takes up what the last step left)
    float4 r[NL];
    r[0] = adjoint<0, K>(s);
    if constexpr (NL > 1) r[1] = adjoint<1, K>(s);
    const int p = e - G::OA(0);
    if (p >= G::A() && p < M + G::A()) st4(rout + (size_t)(p & (M - 1)) * M, r[0]);
#pragma unroll
    for (int j = 0; j + 1 < NL; ++j) q[j] = sub4(r[j + 1], ui[j]);
    const int oc = e - G::OFF(NL - 1);
    if (oc < M) {
      float4 cn[NL], nu[NL];
      analysis<0, K>(s, e, &cn[0], &nu[0]);
      if constexpr (NL > 1) analysis<1, K>(s, e, &cn[1], &nu[1]);
      const float4 uj = dual4(u[NL], cn[NL - 1], k, rho);
      if (oc >= 0) st4(U + (size_t)NL * plane + (size_t)oc * M, uj);
      q[NL - 1] = sub4(uj, nu[NL - 1]);
#pragma unroll
      for (int j = 1; j < NL; ++j) x[j] = cn[j - 1];
    } else {
      q[NL - 1] = sub4(u[NL], u[NL - 1]);
    }
    x[0] = xn;
#pragma unroll
    for (int j = 0; j <= NL; ++j) u[j] = un[j];
#pragma unroll
    for (int j = 0; j < NL; ++j) {
      ui[j] = uin[j];
      uc[j] = ucn[j];
    }
  }
};

// Warp `unit`: sub-image unit % 4^j1 of channel unit / 4^j1.
template <int NL>
__global__ void __launch_bounds__(32 * kCoarseWarps)
k_coarse_m(int n, int J, int j1, int units, const float* c_in, float* r_out, float* U, float k, float rho) {
  using G = CoarseM<NL>;
  extern __shared__ __align__(16) float sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int unit = blockIdx.x * kCoarseWarps + warp;
  if (unit >= units) return;
  const size_t P = (size_t)n * n;
  const int l = unit >> (2 * j1), cls = unit & ((1 << (2 * j1)) - 1);
  const size_t at = (size_t)cls * M * M + 4 * lane;
  CoarseWarp<NL> w;
  w.cin = c_in + (size_t)l * P + at;
  w.rout = r_out + (size_t)l * P + at;
  w.U = U + ((size_t)l * (J + 1) + j1) * P + at;
  w.plane = P;
  w.ring = sm + (size_t)warp * G::ROWS * M + 4 * lane;
  w.lane = lane;
  w.k = k;
  w.rho = rho;
  const float4 zero = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
  for (int i = 0; i < 4; ++i) w.ra[i] = w.rb[i] = zero;
#pragma unroll
  for (int i = 0; i < G::ROWS; ++i) st4(w.ring + i * M, zero);
#pragma unroll
  for (int j = 0; j < NL; ++j) w.x[j] = w.q[j] = w.ui[j] = w.uc[j] = w.u[j] = zero;
  w.u[NL] = zero;
  w.x[0] = ldg4(w.cin + (size_t)((-G::A()) & (M - 1)) * M);
  const int steps = M + 2 * G::A() + G::OA(0);
  for (int s = 0; s < steps; s += 4) {
    w.template step<0>(s);
    w.template step<1>(s + 1);
    w.template step<2>(s + 2);
    w.template step<3>(s + 3);
  }
}

}  // namespace march

// One or two levels on 128 x 128 sub-images at the largest split (N = 1024),
// 512 of them (8 channels) at least.  Pass of 1024 x 1024 x L with one level, us,
// block kernel / march: L = 4 197 / 213, 5 254 / 246, 6 276 / 308, 7 300 / 326, 8
// 352 / 332, 9 381 / 395, 10 431 / 423, 12 514 / 489, 16 625 / 564; with two: 4 230
// / 262, 5 301 / 289, 6 324 / 368, 7 352 / 385, 8 414 / 402, 9 450 / 452, 10 511 /
// 481, 12 605 / 543, 16 743 / 621.  Smaller images reach 64 x 64 sub-images and
// their resident kernel with a larger split; at 512 x 512 x 64, J = 4, the
// march at j1 = 2 is the faster wavelet half on its own (0.240 against 0.283
// ms), but hides less of the spectral step beside it (pass 0.515 against 0.483).
bool coarse_march_ok(const Geom& g) {
  const int NL = g.J - g.j1;
  return g.vec && g.gen == 1 && g.j1 == 3 && (g.n >> 3) == march::M && (NL == 1 || NL == 2) && g.L * 64 >= 512;
}

template <int NL>
static cudaError_t coarse_march(const Geom& g, const float* c_in, float* r_out, float* U, float k, float rho,
                                cudaStream_t s) {
  const int units = g.L << (2 * g.j1);
  march::k_coarse_m<NL><<<(units + march::kCoarseWarps - 1) / march::kCoarseWarps, 32 * march::kCoarseWarps,
                          march::CoarseM<NL>::SMEM, s>>>(g.n, g.J, g.j1, units, c_in, r_out, U, k, rho);
  return cudaGetLastError();
}

cudaError_t launch_coarse_march(const Geom& g, const float* c_in, float* r_out, float* U, float k, float rho,
                                cudaStream_t s) {
  return g.J - g.j1 == 1 ? coarse_march<1>(g, c_in, r_out, U, k, rho, s) : coarse_march<2>(g, c_in, r_out, U, k, rho, s);
}

}  // namespace muffin
