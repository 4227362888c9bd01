// Warm-start network: six zero-padded 3x3x3 convolution layers over the
// cube (1 -> 32 -> 32 -> 32 -> 32 -> 32 -> K feature maps, K <= 8), its
// loss, its gradients and Adam, all in bfloat16 with float32 accumulation.
// Output map 0 predicts the cube X of Algorithm 1, maps 1 .. K-1 further
// fields of its state (the planes of the wavelet dual U).
//
// Feature maps are [nz][ny][nx][32] bfloat16 (64 bytes per voxel).  The
// tensor-core kernels (below) march tiles of 1 x 16 x 8 voxels along the
// channel axis.  The CUDA-core kernels of the first and last layers work on output tiles
// of 2 x 8 x 16 voxels (channel, row, column) whose scalar inputs, with a
// one-voxel halo (4 x 10 x 18, zero outside the cube: the zero padding of the
// layers), are staged in shared memory.
//
// The 32 -> 32 layers are implicit GEMMs on the tensor cores, bfloat16 in,
// float32 accumulate:
//   forward      z[p][co]  = sum_tap sum_ci a[p + d(tap)][ci] W[tap][co][ci]
//                 (M = voxels, N = co, K = 27 taps x 32 ci), tcgen05.mma with the
//                 accumulator in tensor memory,
//   input grad   da[p][ci] = sum_tap sum_co dz[p - d(tap)][co] W[tap][co][ci],
//                 the same kernel on the flipped, transposed weights,
//   weight grad  dW[tap][co][ci] = sum_p dz[p][co] a[p + d(tap)][ci]
//                 (M = (row offset, ci), N = (channel offset, co), K = voxels), tcgen05.mma
//                 with the accumulators resident in tensor memory for the CTA's whole run.
// The last layer's forward (prediction, or the loss and its gradient d6) is
// the forward kernel with 16 columns an output (weights of maps K .. 15 zero).
// Its gradients, whose operand d6 is float32, and the 1 -> 32 layer (27
// multiply-adds per voxel and output) run on the CUDA cores.  Every reduction over voxels is a per-block partial sum
// followed by a fixed-order sum: results do not depend on scheduling.
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <string>

#include "device.cuh"
#include "exact_sum.cuh"
#include "muffin.h"
#include "muffin_net.h"

namespace mnet {

using bf16 = __nv_bfloat16;
using bf162 = __nv_bfloat162;

constexpr int C = 32;                        // features of the hidden layers
constexpr int NTAP = 27;
constexpr int TZ = 2, TY = 8, TX = 16;       // output tile (channel, row, column)
constexpr int TV = TZ * TY * TX;             // 256 voxels
constexpr int HZ = TZ + 2, HY = TY + 2, HX = TX + 2;
constexpr int HV = HZ * HY * HX;             // 720 voxels with halo
constexpr int ROWB = C * 2;                  // 64 bytes per voxel of a map
constexpr int WMID = NTAP * C * C;           // 27648 weights of a 32 -> 32 layer
constexpr int kMaxOut = 8;                   // output maps of the last layer, at most
constexpr int kMaxPart = 512;                // cap of per-block partial slots (weight gradients)
constexpr int kMaxLossPart = 1024;


struct Dims {
  int nz, ny, nx;
  int tx, ty, tz;   // tiles along each axis
  int ntiles;
  long long nvox;
};

inline Dims make_dims(int nz, int ny, int nx) {
  Dims d;
  d.nz = nz; d.ny = ny; d.nx = nx;
  d.tx = (nx + TX - 1) / TX; d.ty = (ny + TY - 1) / TY; d.tz = (nz + TZ - 1) / TZ;
  d.ntiles = d.tx * d.ty * d.tz;
  d.nvox = (long long)nz * ny * nx;
  return d;
}

// ------------------------------------------------------------------ helpers

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(src_bytes) : "memory");
}

__device__ __forceinline__ void cp_async_wait_all() {
  asm volatile("cp.async.commit_group;\ncp.async.wait_group 0;\n" ::: "memory");
}

__device__ __forceinline__ void tile_origin(int tile, const Dims& d, int& z0, int& y0, int& x0) {
  const int tx = tile % d.tx;
  const int r = tile / d.tx;
  x0 = tx * TX;
  y0 = (r % d.ty) * TY;
  z0 = (r / d.ty) * TZ;
}

__device__ __forceinline__ bool inside(const Dims& d, int z, int y, int x) {
  return (unsigned)z < (unsigned)d.nz && (unsigned)y < (unsigned)d.ny && (unsigned)x < (unsigned)d.nx;
}

__device__ __forceinline__ size_t vox(const Dims& d, int z, int y, int x) {
  return ((size_t)z * d.ny + y) * d.nx + x;
}

// Scalar field halo (float32 cube or bfloat16 single-feature map) into s[h], zero outside.
template <typename T>
__device__ __forceinline__ void load_scalar_halo(float* s, const T* __restrict__ g, const Dims& d, int z0, int y0,
                                                 int x0) {
  for (int h = threadIdx.x; h < HV; h += blockDim.x) {
    const int hx = h % HX, t = h / HX, hy = t % HY, hz = t / HY;
    const int gz = z0 - 1 + hz, gy = y0 - 1 + hy, gx = x0 - 1 + hx;
    float v = 0.f;
    if (inside(d, gz, gy, gx)) v = static_cast<float>(g[vox(d, gz, gy, gx)]);
    s[h] = v;
  }
}

__device__ __forceinline__ void unpack8(uint4 q, float* f) {
  const bf162* p = reinterpret_cast<const bf162*>(&q);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const float2 t = __bfloat1622float2(p[e]);
    f[2 * e] = t.x;
    f[2 * e + 1] = t.y;
  }
}

__device__ __forceinline__ uint4 pack8(const float* f) {
  uint4 q;
  bf162* p = reinterpret_cast<bf162*>(&q);
#pragma unroll
  for (int e = 0; e < 4; ++e) p[e] = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
  return q;
}

// ------------------------------------------------------------------ 32 -> 32 layers on the tensor cores

// Epilogues of the tcgen05 layer: the 32 -> 32 layers (bias + ReLU, bias, or
// the ReLU mask of an input gradient) and the last layer (prediction, or loss).
enum { EPI_RELU = 0, EPI_BIAS = 1, EPI_MASK = 2, EPI_PRED = 3, EPI_LOSS = 4 };

// Per-output-map constants of the last layer (at most kMaxOut maps), by value.
struct Lam {
  float v[kMaxOut];
};

// Operands of the last layer's epilogues (unused by the 32 -> 32 layers).
struct LastArgs {
  int K;                      // output maps
  Lam lam;                    // loss weights
  const float* s;             // input scale (device scalar)
  const float* tx;            // EPI_LOSS: target cube [V]
  const bf16* taux;           // EPI_LOSS: target fields [nz][K-1][ny][nx]
  float* d6;                  // EPI_LOSS: loss gradient [V][K]
  double* lpart;              // EPI_LOSS: per-CTA partial sums [grid][K+1]
  float* out_x;               // EPI_PRED: cube [V]
  float* out_aux;             // EPI_PRED: fields [nz][K-1][ny][nx]
};

// ------------------------------------------------------------------ 32 -> 32 layers on tcgen05 (UMMA), marching along z
//
// A CTA walks output tiles of 128 voxels (one channel, 16 rows, 8 columns)
// along the channel axis z, column of tiles after column of tiles.  Input
// planes (the 18 x 10 halo of one channel) arrive one by one; plane i feeds
// the three outputs z = i-1, i, i+1 with its taps kz = 2, 1, 0.  Their
// accumulators D[128 voxels][32 features] lie side by side in tensor memory,
// and the weights of the three kz side by side in shared memory, so one
// tcgen05.mma (kind::f16, bfloat16 A and B, float32 D, M = 128, K = 16) with
// N = 96 serves all three: 18 MMAs a tile (9 shifts in the plane x 2 steps of
// K) where one per tap and output makes 54 of N = 32.  An MMA of N = 32 takes
// as long as one of N = 96 (57 and 60 cycles measured): its time is the read
// of the 4 KB A operand.  Every output still sums its 27 taps in the order kz,
// ky, kx, K step.  The last layer, whose epilogue writes the prediction or the
// loss terms, runs with 16 columns an output (N = 48).
//
// Eight accumulators (256 of the 512 columns: two CTAs per SM) form a ring; an
// MMA whose outputs run over its end is issued in two parts, and the first MMA
// into a new accumulator is issued apart, without the accumulate flag.
//
// Roles: warps 4-7 load planes with 16-byte cp.async (zero fill outside the
// cube: the zero padding of the layer) into a ring of shared-memory slots,
// [chunk of 8 features][row][column][16 B] (the canonical K-major layout
// without swizzle: 8 voxels of a row are one core matrix in every shifted
// window; the chunk pitch of 2976 B spreads the chunks over the banks); warp
// 8 issues the MMAs; warps 0-3 drain the accumulators.  (TMA boxes of 16-byte
// rows, which this layout needs, move one 16-byte piece per two cycles and
// fetch a 32-byte sector for each: they took 4300 of the 5150 cycles per tile
// of a kernel that loaded each tile's halo so.)
// Weights are [shift][chunk][2 - kz][co][16 B] (next 8 outputs 128 B, next 8
// inputs 1536 B), loaded once per CTA.
//
// Every wait is bounded: a warp that gives up (all of its lanes together:
// warp_wait) records it in g_tc_timeouts and leaves, the others run into their
// own bounds, and the CTA waits for its copies and MMAs in flight (at the full
// bound) before it frees its tensor memory.
constexpr int U_TY = 16, U_TX = 8;                          // output tile: 16 rows x 8 columns, one channel
constexpr int U_HY = U_TY + 2, U_HX = U_TX + 2;             // 18 x 10 halo of a plane
constexpr int Z_CH = 2976;                                  // chunk pitch of a plane slot (180 voxels x 16 B, padded)
constexpr int Z_PLANE = 4 * Z_CH;                           // 11904
constexpr int Z_NS = 4;                                     // plane slots
constexpr int Z_PIECES = U_HY * U_HX * 4;                   // 16-byte pieces of a plane: 720
constexpr int Z_RING = 8;                                   // accumulators
constexpr int kLastN = 16;                                  // columns of an output of the last layer (K <= 8 maps used)
template <int EPI> __host__ __device__ constexpr int epi_n() { return EPI >= EPI_PRED ? kLastN : C; }
// weights: 55296 B (N = 32), 27648 B (N = 16); then the mbarriers and the TMEM address slot; alignment slack
__host__ __device__ constexpr int u_w(int no) { return NTAP * 4 * no * 16; }
__host__ __device__ constexpr int u_bar(int no) { return Z_NS * Z_PLANE + u_w(no); }
__host__ __device__ constexpr int conv05_smem(int no) { return u_bar(no) + 256 + 128; }
// D f32, A/B bf16, both K-major, N = no, M = 128
__host__ __device__ constexpr uint32_t idesc_bf16(int no) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(no >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}
constexpr long long kWaitLimit = 1LL << 20;   // polls; each may suspend for a bounded time

__device__ int g_tc_timeouts;
// Poll bound of the pipeline waits (settable through muffin_net_set_wait_limit).
// The drain waits after a give-up keep the full bound kWaitLimit, so that no
// copy or MMA lands in shared or tensor memory after the CTA has left.
__device__ long long g_wait_polls = kWaitLimit;

__device__ __forceinline__ uint64_t umma_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= (uint64_t)1 << 46;   // descriptor version of sm_100 and later; swizzle mode 0 (none)
  return d;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

__device__ __forceinline__ bool mbar_wait_n(uint32_t bar, uint32_t parity, long long limit) {
  uint32_t done = 0;
  for (long long it = 0; it < limit && !done; ++it) {
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
  }
  return done != 0;
}
// Pipeline wait: gives up after `polls` polls, g_wait_polls as the kernel read
// it once at its start (read at each wait, the load's latency, some 700 cycles,
// stood in front of every poll).
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, long long polls) {
  return mbar_wait_n(bar, parity, polls);
}
// The same for a whole warp, as one decision: its lanes poll on their own and
// may see the bound run out differently, and a lane that left alone would let
// the others run the warp's aligned tcgen05 loads, or wait in a full-mask vote,
// without it.  The vote also brings the lanes together again.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, long long polls) {
  return __all_sync(0xffffffffu, mbar_wait_n(bar, parity, polls));
}
// drain wait after a give-up: the full bound
__device__ __forceinline__ bool mbar_drain(uint32_t bar, uint32_t parity) { return mbar_wait_n(bar, parity, kWaitLimit); }

__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// The run of output tiles of this CTA: tiles are numbered column by column
// (z fastest) and split evenly.
struct Runs {
  long long at, end;
  __device__ __forceinline__ Runs(int ncol, int nz) {
    const long long total = (long long)ncol * nz;
    at = total * blockIdx.x / gridDim.x;
    end = total * (blockIdx.x + 1) / gridDim.x;
  }
  // input planes of the whole run: each stretch reads one before and one after its tiles
  __device__ __forceinline__ int planes(int nz) const {
    return at < end ? (int)(end - at + 2 * ((end - 1) / nz - at / nz + 1)) : 0;
  }
  // next stretch za .. zb-1 of one column; false at the end
  __device__ __forceinline__ bool next(int nz, int& col, int& za, int& zb) {
    if (at >= end) return false;
    col = (int)(at / nz);
    za = (int)(at % nz);
    const long long left = end - at;
    zb = left < nz - za ? za + (int)left : nz;
    at += zb - za;
    return true;
  }
};

template <int EPI>
__global__ void __launch_bounds__(288, 2)
k_conv_tc05(const bf16* __restrict__ in, const bf16* __restrict__ wk, const float* __restrict__ bias,
            const bf16* __restrict__ mask, bf16* __restrict__ out, Dims d, int tiles_x, int tiles_y, LastArgs la) {
  constexpr int NO = epi_n<EPI>();
  constexpr bool kLast = EPI >= EPI_PRED;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ double s_red[32];
  const uint32_t s0 = (smem_u32(smem) + 127u) & ~127u;
  const uint32_t s_w = s0 + Z_NS * Z_PLANE;
  const uint32_t s_full = s0 + u_bar(NO);          // plane loaded, per slot (128 loader threads)
  const uint32_t s_free = s_full + 8 * Z_NS;       // plane's MMAs done, per slot
  const uint32_t s_done = s_free + 8 * Z_NS;       // output complete, per accumulator
  const uint32_t s_read = s_done + 8 * Z_RING;     // accumulator read (128 epilogue threads)
  const uint32_t s_fin = s_read + 8 * Z_RING;      // everything the issuer started has finished
  const uint32_t s_tm = s_fin + 8;                 // TMEM address written by tcgen05.alloc
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // weights [tap][co][ci] -> [shift][chunk][2 - kz][co][16 B], once per CTA
  for (int i = threadIdx.x; i < NTAP * NO * 4; i += blockDim.x) {
    const int c = i & 3, co = (i >> 2) % NO, t = i / (4 * NO), sh = t % 9, kz = t / 9;
    cp_async16(s_w + (uint32_t)((((sh * 4 + c) * 3 + 2 - kz) * NO + co) * 16), wk + (t * NO + co) * C + c * 8, 16);
  }
  cp_async_wait_all();
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // generic-proxy writes, read by the MMA
  if (threadIdx.x == 0) {
    for (int b = 0; b < Z_NS; ++b) {
      muffin::mbar_init(s_full + 8 * b, 128);
      muffin::mbar_init(s_free + 8 * b, 1);
    }
    for (int b = 0; b < Z_RING; ++b) {
      muffin::mbar_init(s_done + 8 * b, 1);
      muffin::mbar_init(s_read + 8 * b, 128);
    }
    muffin::mbar_init(s_fin, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 256;" ::"r"(s_tm) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  uint32_t tmem;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem) : "r"(s_tm) : "memory");

  const long long polls = *(volatile long long*)&g_wait_polls;
  Runs runs(tiles_x * tiles_y, d.nz);
  int col, za, zb;
  bool ok = true;
  // EPI_LOSS: sums of lam r^2 and of r of each map
  double l2 = 0.0, lsum[EPI == EPI_LOSS ? kMaxOut : 1] = {};

  if (warp >= 4 && warp < 8) {
    // ---------------- loaders: planes za-1 .. zb of each stretch, two planes in flight behind the newest
    constexpr int NP = (Z_PIECES + 127) / 128;
    const int tid = threadIdx.x - 128;
    const unsigned char* base = reinterpret_cast<const unsigned char*>(in);
    const size_t pitch = (size_t)d.ny * d.nx * ROWB;
    int np = 0;                                     // planes issued so far
    auto landed = [&](int p) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(s_full + 8 * (p % Z_NS));
    };
    while (ok && runs.next(d.nz, col, za, zb)) {
      const int x0 = (col % tiles_x) * U_TX, y0 = (col / tiles_x) * U_TY;
      uint32_t off[NP], dst[NP];
      bool in_xy[NP];
#pragma unroll
      for (int i = 0; i < NP; ++i) {
        const int id = tid + 128 * i, c = id & 3, v = id >> 2, hx = v % U_HX, hy = v / U_HX;
        const int gy = y0 - 1 + hy, gx = x0 - 1 + hx;
        in_xy[i] = (unsigned)gy < (unsigned)d.ny && (unsigned)gx < (unsigned)d.nx;
        off[i] = in_xy[i] ? ((uint32_t)gy * (uint32_t)d.nx + (uint32_t)gx) * ROWB + c * 16 : 0u;
        dst[i] = (uint32_t)(c * Z_CH + v * 16);
      }
      for (int z = za - 1; z <= zb; ++z) {
        const int slot = np % Z_NS;
        if (!warp_wait(s_free + 8 * slot, (uint32_t)(np / Z_NS & 1) ^ 1u, polls)) { ok = false; break; }
        const bool in_z = (unsigned)z < (unsigned)d.nz;
        const unsigned char* pl = base + (in_z ? (size_t)z * pitch : 0);
        const uint32_t sp = s0 + slot * Z_PLANE;
#pragma unroll
        for (int i = 0; i < NP; ++i)
          if (tid + 128 * i < Z_PIECES) cp_async16(sp + dst[i], pl + off[i], in_z && in_xy[i] ? 16 : 0);
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (np >= 2) {
          asm volatile("cp.async.wait_group 2;" ::: "memory");
          landed(np - 2);
        }
        ++np;
      }
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (ok) {
      if (np >= 2) landed(np - 2);
      if (np >= 1) landed(np - 1);
    }
  } else if (warp == 8) {
    // ---------------- issuer
    int np = 0, no = 0;                             // planes taken, outputs finished before this stretch
    const uint64_t wd0 = umma_desc(s_w, 3 * NO * 16, 8 * 16);
    // MMA of shift / K step (its offsets within the plane and the weights) into nb accumulators from ring block
    // blk on, weight blocks from b0 on
    auto mma = [&](uint64_t ad, uint64_t wd, int blk, int nb, int b0, uint32_t accum) {
      asm volatile(
          "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
          "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)(blk * NO)),
          "l"(ad), "l"(wd + (uint64_t)(b0 * NO)), "r"(idesc_bf16(nb * NO)), "r"(accum)
          : "memory");
    };
    while (lane == 0 && ok && runs.next(d.nz, col, za, zb)) {
      const int n = zb - za;
      for (int i = 0; i < n + 2; ++i) {             // plane za - 1 + i feeds outputs i-2 .. i of the stretch
        const int slot = np % Z_NS;
        const int lo = i < 2 ? 0 : i - 2, hi = i < n ? i : n - 1;
        if (!mbar_wait(s_full + 8 * slot, (uint32_t)(np / Z_NS & 1), polls)) { ok = false; break; }
        if (i < n) {                                // output i starts here: its accumulator must have been read
          const int o = no + i;
          if (!mbar_wait(s_read + 8 * (o % Z_RING), (uint32_t)(o / Z_RING & 1) ^ 1u, polls)) { ok = false; break; }
        }
        tc_fence_after();
        // outputs lo .. hi as one or two runs of the ring
        const int blk = (no + lo) % Z_RING, nb = hi - lo + 1, b0 = lo - (i - 2);
        const int n1 = blk + nb > Z_RING ? Z_RING - blk : nb;
        const uint64_t ad0 = umma_desc(s0 + slot * Z_PLANE, Z_CH, U_HX * 16);
        // first shift and step: a new output's accumulator is overwritten
        if (i < n) {
          if (nb > 1) {
            const int m1 = n1 < nb ? n1 : nb - 1;
            mma(ad0, wd0, blk, m1, b0, 1u);
            if (nb - 1 > m1) mma(ad0, wd0, 0, nb - 1 - m1, b0 + m1, 1u);
          }
          mma(ad0, wd0, (no + i) % Z_RING, 1, 2, 0u);
        } else {
          mma(ad0, wd0, blk, n1, b0, 1u);
          if (n1 < nb) mma(ad0, wd0, 0, nb - n1, b0 + n1, 1u);
        }
#pragma unroll
        for (int q = 1; q < 18; ++q) {
          const int sh = q >> 1, kk = q & 1;
          const uint64_t ad = ad0 + (uint64_t)((sh / 3) * U_HX + sh % 3 + kk * 2 * (Z_CH / 16));
          const uint64_t wd = wd0 + (uint64_t)((sh * 4 + kk * 2) * 3 * NO);
          mma(ad, wd, blk, n1, b0, 1u);
          if (n1 < nb) mma(ad, wd, 0, nb - n1, b0 + n1, 1u);
        }
        tc_commit(s_free + 8 * slot);
        ++np;
        if (i >= 2) tc_commit(s_done + 8 * ((no + i - 2) % Z_RING));
      }
      no += n;
    }
    if (lane == 0) tc_commit(s_fin);
    __syncwarp();
  } else if (warp < 4) {
    // ---------------- epilogue: row m = 32 warp + lane of D is voxel (y0 + m / 8, x0 + m % 8)
    float bn[NO];
#pragma unroll
    for (int c = 0; c < NO; ++c) bn[c] = (EPI != EPI_MASK && bias && (!kLast || c < la.K)) ? bias[c] : 0.f;
    // last layer: input scale; factors of the loss gradient
    const float sc = kLast ? *la.s : 1.f;
    const float inv_sc = 1.0f / sc;
    float gk[EPI == EPI_LOSS ? kMaxOut : 1];
    if constexpr (EPI == EPI_LOSS) {
#pragma unroll
      for (int k = 0; k < kMaxOut; ++k) gk[k] = (float)(2.0 / (double)d.nvox * la.lam.v[k]);
    }
    const size_t plane = (size_t)d.ny * d.nx;
    const int m = warp * 32 + lane;
    int no = 0;
    while (ok && runs.next(d.nz, col, za, zb)) {
      const int x = (col % tiles_x) * U_TX + (m & 7), y = (col / tiles_x) * U_TY + (m >> 3);
      for (int z = za; z < zb; ++z, ++no) {
        const int acc = no % Z_RING;
        // the loss's targets, loaded while the tile's MMAs run
        float tk[EPI == EPI_LOSS ? kMaxOut : 1];
        if constexpr (EPI == EPI_LOSS) {
          if (inside(d, z, y, x)) {
            tk[0] = la.tx[vox(d, z, y, x)];
            const bf16* ta = la.taux + (size_t)z * (la.K - 1) * plane + (size_t)y * d.nx + x;
#pragma unroll
            for (int k = 1; k < kMaxOut; ++k)
              if (k < la.K) tk[k] = __bfloat162float(ta[(size_t)(k - 1) * plane]);
          }
        }
        if (!warp_wait(s_done + 8 * acc, (uint32_t)(no / Z_RING & 1), polls)) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem + (uint32_t)(acc * NO) + ((uint32_t)(warp * 32) << 16);
        if constexpr (!kLast) {
          uint32_t r[C];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
              "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
                "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
                "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          tc_fence_before();
          mbar_arrive(s_read + 8 * acc);
          if (inside(d, z, y, x)) {
            const size_t base = vox(d, z, y, x) * C;
            float v[C];
#pragma unroll
            for (int c = 0; c < C; ++c) v[c] = __uint_as_float(r[c]);
            if (EPI == EPI_MASK) {
              if (mask) {
                const uint4* mp = reinterpret_cast<const uint4*>(mask + base);
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  float mf[8];
                  unpack8(mp[q], mf);
#pragma unroll
                  for (int e = 0; e < 8; ++e)
                    if (!(mf[e] > 0.f)) v[8 * q + e] = 0.f;
                }
              }
            } else {
#pragma unroll
              for (int c = 0; c < C; ++c) {
                v[c] += bn[c];
                if (EPI == EPI_RELU) v[c] = fmaxf(v[c], 0.f);
              }
            }
            uint4* o = reinterpret_cast<uint4*>(out + base);
#pragma unroll
            for (int q = 0; q < 4; ++q) o[q] = pack8(v + 8 * q);
          }
        } else {
          // last layer: z_k = D[m][k] + b_k for the K maps (columns K .. 15 hold zero weights)
          uint32_t r[kLastN];
          asm volatile(
              "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
              : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
                "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
              : "r"(taddr));
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          tc_fence_before();
          mbar_arrive(s_read + 8 * acc);
          if (inside(d, z, y, x)) {
            const int K = la.K;
            const size_t v = vox(d, z, y, x);
            const size_t a0 = ((size_t)z * (K > 1 ? K - 1 : 1)) * plane + (size_t)y * d.nx + x;
#pragma unroll
            for (int k = 0; k < kMaxOut; ++k) {
              if (k < K) {
                const float zk = __uint_as_float(r[k]) + bn[k];
                if constexpr (EPI == EPI_LOSS) {
                  const float rk = zk - (k == 0 ? tk[0] * inv_sc : tk[k]);
                  la.d6[v * K + k] = gk[k] * rk;
                  l2 += (double)la.lam.v[k] * rk * rk;
                  lsum[k] += rk;
                } else {
                  if (k == 0) la.out_x[v] = fmaxf(sc * zk, 0.f);
                  else la.out_aux[a0 + (size_t)(k - 1) * plane] = fminf(fmaxf(zk, -1.f), 1.f);
                }
              }
            }
          }
        }
      }
    }
  }
  const bool fin = mbar_drain(s_fin, 0);   // every copy and MMA issued, also after a give-up: TMEM is freed below
  tc_fence_before();
  if (__syncthreads_or(!ok || !fin) && threadIdx.x == 0) atomicAdd(&g_tc_timeouts, 1);
  tc_fence_after();
  __syncwarp();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 256;" ::"r"(tmem) : "memory");
  if constexpr (EPI == EPI_LOSS) {
    // lpart[block] = (sum_k lam_k sum_p r_k^2, sum_p r_0, ..., sum_p r_{K-1}), fixed order
    const double t2 = muffin::block_sum(l2, s_red);
    if (threadIdx.x == 0) la.lpart[(size_t)blockIdx.x * (la.K + 1)] = t2;
#pragma unroll
    for (int k = 0; k < kMaxOut; ++k) {
      if (k >= la.K) break;
      __syncthreads();
      const double t = muffin::block_sum(lsum[k], s_red);
      if (threadIdx.x == 0) la.lpart[(size_t)blockIdx.x * (la.K + 1) + 1 + k] = t;
    }
  }
}

// ------------------------------------------------------------------ 32 -> 32 weight gradient on tcgen05, marching along z
//
// dW[tap][co][ci] = sum_p dz[p][co] a[p + d(tap)][ci] as tensor-core products
// D[m][n] += A[m][k] B[k][n] with k = voxel of a tile of one channel,
// m = (ky, ci) and n = (2 - kz, co): the plane zi of a is multiplied with the
// dz planes zi - 1, zi, zi + 1 at once (kz = 2, 1, 0), so one accumulator of
// 128 x 96 per kx holds the nine row and channel offsets of its taps (rows
// 96..127, "ky = 3", are computed and dropped).  The three accumulators (288
// columns) stay in tensor memory; every `flush` planes their sums are added to
// float32 sums in shared memory, rounded to nearest, and they start over, since
// the tensor core adds with truncation: a run of 1700 additions of one sign
// loses 8e-5 of its sum (wgrad_flush has the rule).  24 MMAs of N = 96 per tile
// replace 72 of N = 32; an MMA takes as long either way (the read of its A
// operand).
//
// Both operands are MN-major (M or N contiguous: the 8 features of a chunk),
// canonical layout without swizzle: core matrices of 8 voxels x 16 bytes.  A
// plane of a with its halo (rows y0-1 .. y0+17, the last one only feeding the
// dropped rows) is [row][chunk][column][16 B]: the next 8 rows of m (next
// chunk, or next ky after four) are 160 B apart, the next 8 voxels of k (next
// row) 640 B.  The dz tiles of eight channels form a ring
// [row][ring slot][chunk][column][16 B], so that consecutive channels continue
// n: next 8 of n 128 B, next 8 voxels 4096 B; MMAs that run over the ring's end
// are issued in two parts.
//
// Roles: warps 4-7 load with 16-byte cp.async (zero fill outside the cube),
// warp 8 issues the MMAs, warps 0-3 sum the dz tiles into the bias gradient
// as they land and store the sums at the end.  One CTA per SM.  Every wait is
// bounded; a CTA that gives up records it in g_tc_timeouts, waits (bounded) for
// its copies and MMAs in flight, writes nothing and frees its tensor memory.
constexpr int WG_HY = U_TY + 3;                        // 19 rows (one extra for the dropped ones)
constexpr int WG_CH = U_HX * 16;                       // chunk pitch 160 B
constexpr int WG_ROW = 4 * WG_CH;                      // row pitch 640 B
constexpr int WG_A = WG_HY * WG_ROW;                   // 12160 B
constexpr int WG_NS = 4;                               // slots of a planes
constexpr int WG_R = 8;                                // ring of dz tiles (more than WG_NS + 2)
constexpr int WG_DROW = WG_R * 4 * U_TX * 16;          // row pitch of the ring 4096 B
constexpr int WG_B = U_TY * WG_DROW;                   // 65536 B
constexpr int WG_BAR = WG_NS * WG_A + WG_B;            // full, free, fin, TMEM slot
constexpr int WG_SUM = 3 * 3 * C * 96 * 4;              // flushed sums, 110592 B
// more than half an SM: one CTA holds all of the tensor memory
constexpr int wgrad05_smem = WG_BAR + 256 + 128 + WG_SUM;
static_assert(wgrad05_smem + 4096 <= muffin::kMaxDynSmem, "weight gradient shared memory");
constexpr int WG_N = 3 * C;
// D f32, A/B bf16, both MN-major, N = n, M = 128
__host__ __device__ constexpr uint32_t idesc_wgrad(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(128 >> 4) << 24);
}

__global__ void __launch_bounds__(288, 1)
k_wgrad_tc05(const bf16* __restrict__ a, const bf16* __restrict__ dz, float* __restrict__ part,
             float* __restrict__ bpart, Dims d, int tiles_x, int tiles_y, int flush) {
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ float s_b[128 * 8];
  const uint32_t s0 = (smem_u32(smem) + 127u) & ~127u;
  const uint32_t s_dz = s0 + WG_NS * WG_A;
  const uint32_t s_full = s0 + WG_BAR;          // plane and dz tile loaded, per slot (128 loader threads)
  const uint32_t s_free = s_full + 8 * WG_NS;   // MMAs done and dz summed, per slot (1 + 128 threads)
  const uint32_t s_fin = s_free + 8 * WG_NS;    // every MMA of the CTA finished
  const uint32_t s_stop = s_fin + 8;            // MMAs before a flush finished
  const uint32_t s_go = s_stop + 8;             // accumulators stored and cleared (96 threads)
  const uint32_t s_tm = s_go + 8;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int b = 0; b < WG_NS; ++b) {
      muffin::mbar_init(s_full + 8 * b, 128);
      muffin::mbar_init(s_free + 8 * b, 129);
    }
    muffin::mbar_init(s_fin, 1);
    muffin::mbar_init(s_stop, 1);
    muffin::mbar_init(s_go, 96);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(s_tm) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  uint32_t tmem;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(tmem) : "r"(s_tm) : "memory");
  auto clear = [&] {                            // warps 0-3: this warp's lanes of the accumulators
    const uint32_t ta = tmem + ((uint32_t)(warp * 32) << 16);
    __syncwarp();
    for (int c = 0; c < 3 * WG_N; c += 8)
      asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(ta + (uint32_t)c),
                   "r"(0u)
                   : "memory");
    asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
  };
  // warps 0-2: the sums out of tensor memory, onto this CTA's flushed sums (s_sum), and at the end to part
  float* s_sum = reinterpret_cast<float*>(smem + (s0 - smem_u32(smem)) + WG_BAR + 256);
  auto store = [&](bool add, bool last) {
    // lane = ci, TMEM lanes 32 ky .. 32 ky + 31; columns kx * 96 + (2 - kz) * 32 + co
#pragma unroll 1
    for (int q = 0; q < 18; ++q) {            // (kx, 2 - kz) = q / 2, columns (co) 16 (q % 2) .. + 15
      const int acc = q >> 1, co0 = (q & 1) * 16, kx = acc / 3, kz = 2 - acc % 3;
      uint32_t r[16];
      __syncwarp();
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
            "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(acc * C + co0)));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      float* sp = s_sum + (size_t)(q * 16) * 96 + warp * 32 + lane;
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]) + (add ? sp[j * 96] : 0.f);
      const int tap = kz * 9 + warp * 3 + kx;
      float* pp = part + ((size_t)blockIdx.x * NTAP + tap) * (C * C) + co0 * C + lane;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (last) pp[j * C] = v[j];
        else sp[j * 96] = v[j];
      }
    }
  };
  bool flushed = false;
  if (warp < 4) clear();                        // accumulators start at zero
  tc_fence_before();
  __syncthreads();
  tc_fence_after();

  const long long polls = *(volatile long long*)&g_wait_polls;
  Runs runs(tiles_x * tiles_y, d.nz);
  const int planes = runs.planes(d.nz);         // no flush after the last one: the sums leave then anyway
  int col, za, zb;
  bool ok = true;
  float bacc[8];
#pragma unroll
  for (int e = 0; e < 8; ++e) bacc[e] = 0.f;

  if (warp >= 4 && warp < 8) {
    // ---------------- loaders: step i of a stretch brings plane za - 1 + i of a and dz tile za + i
    constexpr int NA = (WG_HY * U_HX * 4 + 127) / 128, ND = U_TY * U_TX * 4 / 128;
    const int tid = threadIdx.x - 128;
    const unsigned char *pa = reinterpret_cast<const unsigned char*>(a), *pd = reinterpret_cast<const unsigned char*>(dz);
    const size_t pitch = (size_t)d.ny * d.nx * ROWB;
    int np = 0, no = 0;
    auto landed = [&](int p) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      mbar_arrive(s_full + 8 * (p % WG_NS));
    };
    while (ok && runs.next(d.nz, col, za, zb)) {
      const int x0 = (col % tiles_x) * U_TX, y0 = (col / tiles_x) * U_TY, n = zb - za;
      uint32_t aoff[NA], adst[NA], doff[ND], ddst[ND];
      bool ain[NA], din[ND];
#pragma unroll
      for (int i = 0; i < NA; ++i) {
        const int id = tid + 128 * i, c = id & 3, v = id >> 2, hx = v % U_HX, hy = v / U_HX;
        const int gy = y0 - 1 + hy, gx = x0 - 1 + hx;
        ain[i] = (unsigned)gy < (unsigned)d.ny && (unsigned)gx < (unsigned)d.nx;
        aoff[i] = ain[i] ? ((uint32_t)gy * (uint32_t)d.nx + (uint32_t)gx) * ROWB + c * 16 : 0u;
        adst[i] = (uint32_t)(hy * WG_ROW + c * WG_CH + hx * 16);
      }
#pragma unroll
      for (int i = 0; i < ND; ++i) {
        const int id = tid + 128 * i, x = id & 7, c = (id >> 3) & 3, y = id >> 5;
        const int gy = y0 + y, gx = x0 + x;
        din[i] = gy < d.ny && gx < d.nx;
        doff[i] = din[i] ? ((uint32_t)gy * (uint32_t)d.nx + (uint32_t)gx) * ROWB + c * 16 : 0u;
        ddst[i] = (uint32_t)(y * WG_DROW + (c * U_TX + x) * 16);
      }
      for (int i = 0; i < n + 2; ++i) {
        const int slot = np % WG_NS, z = za - 1 + i;
        if (!warp_wait(s_free + 8 * slot, (uint32_t)(np / WG_NS & 1) ^ 1u, polls)) { ok = false; break; }
        const bool in_z = (unsigned)z < (unsigned)d.nz;
        const unsigned char* pl = pa + (in_z ? (size_t)z * pitch : 0);
        const uint32_t sp = s0 + slot * WG_A;
#pragma unroll
        for (int q = 0; q < NA; ++q)
          if (tid + 128 * q < WG_HY * U_HX * 4) cp_async16(sp + adst[q], pl + aoff[q], in_z && ain[q] ? 16 : 0);
        if (i < n) {
          const unsigned char* pz = pd + (size_t)(za + i) * pitch;
          const uint32_t sd = s_dz + (uint32_t)((no + i) % WG_R) * (4 * U_TX * 16);
#pragma unroll
          for (int q = 0; q < ND; ++q) cp_async16(sd + ddst[q], pz + doff[q], din[q] ? 16 : 0);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        if (np >= 2) {
          asm volatile("cp.async.wait_group 2;" ::: "memory");
          landed(np - 2);
        }
        ++np;
      }
      no += n;
    }
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    if (ok) {
      if (np >= 2) landed(np - 2);
      if (np >= 1) landed(np - 1);
    }
  } else if (warp == 8) {
    // ---------------- issuer: plane i of a stretch with the dz tiles lo .. hi = i-2 .. i
    int np = 0, no = 0;
    while (lane == 0 && ok && runs.next(d.nz, col, za, zb)) {
      const int n = zb - za;
      for (int i = 0; i < n + 2; ++i) {
        const int slot = np % WG_NS;
        const int lo = i < 2 ? 0 : i - 2, hi = i < n ? i : n - 1;
        if (!mbar_wait(s_full + 8 * slot, (uint32_t)(np / WG_NS & 1), polls)) { ok = false; break; }
        tc_fence_after();
        const int blk = (no + lo) % WG_R, nb = hi - lo + 1, b0 = lo - (i - 2);
        const int n1 = blk + nb > WG_R ? WG_R - blk : nb;
        const uint64_t ad0 = umma_desc(s0 + slot * WG_A, WG_ROW, WG_CH);
        const uint64_t bd0 = umma_desc(s_dz, WG_DROW, U_TX * 16);
        auto mma = [&](int kx, int rp, int blk0, int cnt, int off) {
          asm volatile(
              "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
              "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)(kx * WG_N + off * C)),
              "l"(ad0 + (uint64_t)(2 * rp * (WG_ROW / 16) + kx)),
              "l"(bd0 + (uint64_t)(2 * rp * (WG_DROW / 16) + blk0 * (4 * U_TX))), "r"(idesc_wgrad(cnt * C)), "r"(1u)
              : "memory");
        };
#pragma unroll 1
        for (int kx = 0; kx < 3; ++kx) {
#pragma unroll
          for (int rp = 0; rp < U_TY / 2; ++rp) {
            mma(kx, rp, blk, n1, b0);
            if (n1 < nb) mma(kx, rp, 0, nb - n1, b0 + n1);
          }
        }
        tc_commit(s_free + 8 * slot);
        ++np;
        if (np % flush == 0 && np < planes) {
          tc_commit(s_stop);
          if (!mbar_wait(s_go, (uint32_t)(np / flush - 1) & 1u, polls)) { ok = false; break; }
          tc_fence_after();
        }
      }
      no += n;
    }
    if (lane == 0) tc_commit(s_fin);
    __syncwarp();
  } else if (warp < 4) {
    // ---------------- bias gradient: this thread's chunk c = tid & 3 ... of voxels tid / 4 + 32 q
    const unsigned char* base = smem + (s_dz - smem_u32(smem));
    const int c = threadIdx.x & 3, v0 = threadIdx.x >> 2;
    int np = 0, no = 0;
    while (ok && runs.next(d.nz, col, za, zb)) {
      const int n = zb - za;
      for (int i = 0; i < n + 2; ++i) {
        const int slot = np % WG_NS;
        if (!warp_wait(s_full + 8 * slot, (uint32_t)(np / WG_NS & 1), polls)) { ok = false; break; }
        if (i < n) {
          const unsigned char* t = base + ((no + i) % WG_R) * (4 * U_TX * 16) + c * U_TX * 16;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int v = v0 + 32 * q;
            float f[8];
            unpack8(*reinterpret_cast<const uint4*>(t + (v >> 3) * WG_DROW + (v & 7) * 16), f);
#pragma unroll
            for (int e = 0; e < 8; ++e) bacc[e] += f[e];
          }
        }
        mbar_arrive(s_free + 8 * slot);
        ++np;
        if (np % flush == 0 && np < planes && warp < 3) {
          if (!warp_wait(s_stop, (uint32_t)(np / flush - 1) & 1u, polls)) { ok = false; break; }
          tc_fence_after();
          store(flushed, false);
          flushed = true;
          clear();
          tc_fence_before();
          mbar_arrive(s_go);
        }
      }
      no += n;
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) s_b[threadIdx.x * 8 + e] = bacc[e];
  }
  const bool fin = mbar_drain(s_fin, 0);   // every MMA issued, also after a give-up: TMEM is freed below
  if (__syncthreads_or(!ok || !fin)) {
    if (threadIdx.x == 0) atomicAdd(&g_tc_timeouts, 1);
  } else {
    tc_fence_after();
    if (warp < 3) {
      store(flushed, true);
    } else if (warp == 3 && bpart) {
      float t = 0.f;                            // feature lane: chunk lane / 8, the 32 threads of that chunk
      for (int v = 0; v < 32; ++v) t += s_b[(v * 4 + (lane >> 3)) * 8 + (lane & 7)];
      bpart[(size_t)blockIdx.x * C + lane] = t;
    }
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  __syncwarp();
  if (warp == 0) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// ------------------------------------------------------------------ first and last layers (CUDA cores)

// a1[p][co] = relu(b[co] + sum_tap a0[p + d(tap)] w[tap][co]).  A thread takes
// the two channels z of one (row, column) of the tile, so that the 32 weights
// of a tap, read once, feed 64 multiply-adds (one channel a thread: as many
// shared-memory reads as groups of four multiply-adds, 0.342 against 0.244 ms
// at 64x256x256).
constexpr int kFirstThreads = TY * TX;
__global__ void __launch_bounds__(kFirstThreads)
k_first_fwd(const bf16* __restrict__ a0, const float* __restrict__ w, const float* __restrict__ b,
            bf16* __restrict__ a1, Dims d) {
  __shared__ __align__(16) float s_w[NTAP * C];
  __shared__ float s_b[C];
  __shared__ float s_h[HV];
  for (int i = threadIdx.x; i < NTAP * C; i += blockDim.x) s_w[i] = w[i];
  if (threadIdx.x < C) s_b[threadIdx.x] = b[threadIdx.x];
  const int tx = threadIdx.x % TX, ty = threadIdx.x / TX;
  for (int tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) {
    int z0, y0, x0;
    tile_origin(tile, d, z0, y0, x0);
    __syncthreads();
    load_scalar_halo(s_h, a0, d, z0, y0, x0);
    __syncthreads();
    float acc[TZ][C];
#pragma unroll
    for (int c = 0; c < C; ++c)
#pragma unroll
      for (int z = 0; z < TZ; ++z) acc[z][c] = s_b[c];
#pragma unroll 1
    for (int t = 0; t < NTAP; ++t) {
      const int kz = t / 9, ky = (t / 3) % 3, kx = t % 3;
      float av[TZ];
#pragma unroll
      for (int z = 0; z < TZ; ++z) av[z] = s_h[((z + kz) * HY + ty + ky) * HX + tx + kx];
      const float4* wr = reinterpret_cast<const float4*>(s_w + t * C);
#pragma unroll
      for (int q = 0; q < C / 4; ++q) {
        const float4 wv = wr[q];
#pragma unroll
        for (int z = 0; z < TZ; ++z) {
          acc[z][4 * q] = fmaf(av[z], wv.x, acc[z][4 * q]);
          acc[z][4 * q + 1] = fmaf(av[z], wv.y, acc[z][4 * q + 1]);
          acc[z][4 * q + 2] = fmaf(av[z], wv.z, acc[z][4 * q + 2]);
          acc[z][4 * q + 3] = fmaf(av[z], wv.w, acc[z][4 * q + 3]);
        }
      }
    }
#pragma unroll
    for (int z = 0; z < TZ; ++z) {
      if (!inside(d, z0 + z, y0 + ty, x0 + tx)) continue;
#pragma unroll
      for (int c = 0; c < C; ++c) acc[z][c] = fmaxf(acc[z][c], 0.f);
      uint4* o = reinterpret_cast<uint4*>(a1 + vox(d, z0 + z, y0 + ty, x0 + tx) * C);
#pragma unroll
      for (int q = 0; q < 4; ++q) o[q] = pack8(acc[z] + 8 * q);
    }
  }
}

// Gradients of the last layer.  Their sums are float32 multiply-adds rounded to
// nearest, which the tensor cores do not offer: as 32 -> 32 gradients of d6 split
// into three bfloat16 parts, exact products and all, they took 0.23 and 0.57 ms
// instead of the times below, but truncated additions left the weight gradient 3
// to 14 times further from 64 bits (31x120x100, five maps: 3.8e-8 -> 3.9e-7) and
// the input gradient with a bias of 1e-6.

// Two float32 multiply-adds in one instruction, each rounded to nearest.
__device__ __forceinline__ void fma2(float2& acc, float2 a, float2 b) {
  unsigned long long* c = reinterpret_cast<unsigned long long*>(&acc);
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(*c) : "l"(*reinterpret_cast<unsigned long long*>(&a)),
      "l"(*reinterpret_cast<unsigned long long*>(&b)));
}

// g5[p][ci] = (a5[p][ci] > 0) * sum_tap sum_k d6[p - d(tap)][k] w[tap][k][ci].
// A thread takes 16 of the features of four voxels (both channels of rows ty and
// ty + 4), so that four 16-byte weight reads, the same for the whole warp, feed
// 64 multiply-adds, and issues them in pairs; d6 lies in planes of one map, whose
// lanes' reads are consecutive.  64x256x256, six maps: 1.58 ms (32 features of one
// voxel a thread, d6 interleaved) -> 1.06, half of the FP32 rate; 1.21 without pairs.
constexpr int LV = TZ * 2;            // voxels of a thread
constexpr int kLastThreads = TV / LV * 2;
template <int K>
__global__ void __launch_bounds__(kLastThreads)
k_last_bwd_data(const float* __restrict__ d6, const float* __restrict__ w, const bf16* __restrict__ a5,
                bf16* __restrict__ g5, Dims d) {
  extern __shared__ __align__(16) float smf[];
  float* s_w = smf;                      // [27][K][32]
  float* s_h = smf + NTAP * K * C;       // [K][HV]
  for (int i = threadIdx.x; i < NTAP * K * C; i += blockDim.x) s_w[i] = w[i];
  const int c0 = threadIdx.x / (TV / LV) * 16, tx = threadIdx.x % TX, ty = threadIdx.x % (TV / LV) / TX;
  for (int tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) {
    int z0, y0, x0;
    tile_origin(tile, d, z0, y0, x0);
    __syncthreads();
    for (int i = threadIdx.x; i < HV * K; i += blockDim.x) {
      const int h = i / K, k = i - h * K;
      const int hx = h % HX, r = h / HX, hy = r % HY, hz = r / HY;
      const int gz = z0 - 1 + hz, gy = y0 - 1 + hy, gx = x0 - 1 + hx;
      s_h[k * HV + h] = inside(d, gz, gy, gx) ? d6[vox(d, gz, gy, gx) * K + k] : 0.f;
    }
    __syncthreads();
    float2 acc[LV][8];                   // voxel v: channel v / 2, row ty + 4 (v % 2)
#pragma unroll
    for (int v = 0; v < LV; ++v)
#pragma unroll
      for (int c = 0; c < 8; ++c) acc[v][c] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int t = 0; t < NTAP; ++t) {
      const int kz = t / 9, ky = (t / 3) % 3, kx = t % 3;
      const float* h = s_h + ((2 - kz) * HY + ty + 2 - ky) * HX + tx + 2 - kx;
#pragma unroll
      for (int k = 0; k < K; ++k) {
        float2 dv[LV];
#pragma unroll
        for (int v = 0; v < LV; ++v) dv[v].x = dv[v].y = h[k * HV + (v / 2 * HY + v % 2 * 4) * HX];
        const float4* wr = reinterpret_cast<const float4*>(s_w + (t * K + k) * C + c0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const float4 wv = wr[q];
#pragma unroll
          for (int v = 0; v < LV; ++v) {
            fma2(acc[v][2 * q], dv[v], make_float2(wv.x, wv.y));
            fma2(acc[v][2 * q + 1], dv[v], make_float2(wv.z, wv.w));
          }
        }
      }
    }
#pragma unroll
    for (int v = 0; v < LV; ++v) {
      const int z = z0 + v / 2, y = y0 + ty + v % 2 * 4, x = x0 + tx;
      if (!inside(d, z, y, x)) continue;
      const size_t at = vox(d, z, y, x) * C + c0;
      const uint4* m = reinterpret_cast<const uint4*>(a5 + at);
      uint4* o = reinterpret_cast<uint4*>(g5 + at);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float mf[8], r[8];
        unpack8(m[q], mf);
#pragma unroll
        for (int e = 0; e < 8; ++e) r[e] = !(mf[e] > 0.f) ? 0.f : e & 1 ? acc[v][4 * q + e / 2].y : acc[v][4 * q + e / 2].x;
        o[q] = pack8(r);
      }
    }
  }
}

// part[b][tap][ci][k] = sum_p d6[p][k] a5[p + d(tap)][ci].  288 threads: thread
// (kz, ky, ci) keeps the three taps kx = 0..2 of its row offset for all K maps in
// registers and walks each tile row along x with a sliding window of three a5
// values, so that one a5 read and the voxel's d6 values (one or two 16-byte reads,
// the same for the whole block) feed 3 K multiply-adds.  64x256x256, six maps:
// 1.55 ms (a 4-byte read for each d6 value, swizzled a5 rows) -> 1.32; two features
// a thread 1.36, with pairs of multiply-adds 1.52.
template <int K> __host__ __device__ constexpr int last_pitch() { return K == 1 ? 1 : K == 2 ? 2 : K <= 4 ? 4 : 8; }
template <int K>
__global__ void __launch_bounds__(288)
k_wgrad_last(const float* __restrict__ d6, const bf16* __restrict__ a5, float* __restrict__ part, Dims d) {
  constexpr int KP = last_pitch<K>();
  extern __shared__ __align__(128) unsigned char smem[];     // a5 halo [HV][32] bfloat16, then d6 [TV][KP]
  const uint32_t sa = smem_u32(smem);
  float* s_d = reinterpret_cast<float*>(smem + HV * ROWB);
  const int ci = threadIdx.x & 31, kzy = threadIdx.x >> 5, kz = kzy / 3, ky = kzy % 3;
  const bf16* s_a = reinterpret_cast<const bf16*>(smem) + ci;
  float acc[3][K];
#pragma unroll
  for (int kx = 0; kx < 3; ++kx)
#pragma unroll
    for (int k = 0; k < K; ++k) acc[kx][k] = 0.f;
  for (int tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) {
    int z0, y0, x0;
    tile_origin(tile, d, z0, y0, x0);
    __syncthreads();
    for (int i = threadIdx.x; i < HV * 4; i += blockDim.x) {
      const int c = i & 3, h = i >> 2;
      const int hx = h % HX, t = h / HX, hy = t % HY, hz = t / HY;
      const int gz = z0 - 1 + hz, gy = y0 - 1 + hy, gx = x0 - 1 + hx;
      const bool ok = inside(d, gz, gy, gx);
      cp_async16(sa + h * ROWB + c * 16, ok ? a5 + vox(d, gz, gy, gx) * C + c * 8 : a5, ok ? 16 : 0);
    }
    for (int i = threadIdx.x; i < TV * K; i += blockDim.x) {
      const int r = i / K, k = i - r * K;
      const int gz = z0 + (r >> 7), gy = y0 + ((r >> 4) & 7), gx = x0 + (r & 15);
      s_d[r * KP + k] = inside(d, gz, gy, gx) ? d6[vox(d, gz, gy, gx) * K + k] : 0.f;
    }
    cp_async_wait_all();
    __syncthreads();
#pragma unroll 1
    for (int row = 0; row < TZ * TY; ++row) {
      const int tz = row >> 3, ty = row & 7;
      const bf16* ar = s_a + ((tz + kz) * HY + ty + ky) * HX * C;   // halo row of this thread's taps
      const float* dr = s_d + row * TX * KP;
      float w0 = __bfloat162float(ar[0]), w1 = __bfloat162float(ar[C]);
#pragma unroll 4
      for (int tx = 0; tx < TX; ++tx) {
        const float w2 = __bfloat162float(ar[(tx + 2) * C]);
        float g[KP];
        if constexpr (KP >= 4) {
#pragma unroll
          for (int q = 0; q < KP / 4; ++q) {
            const float4 v = *reinterpret_cast<const float4*>(dr + tx * KP + 4 * q);
            g[4 * q] = v.x; g[4 * q + 1] = v.y; g[4 * q + 2] = v.z; g[4 * q + 3] = v.w;
          }
        } else {
#pragma unroll
          for (int k = 0; k < KP; ++k) g[k] = dr[tx * KP + k];
        }
#pragma unroll
        for (int k = 0; k < K; ++k) {
          acc[0][k] = fmaf(g[k], w0, acc[0][k]);
          acc[1][k] = fmaf(g[k], w1, acc[1][k]);
          acc[2][k] = fmaf(g[k], w2, acc[2][k]);
        }
        w0 = w1;
        w1 = w2;
      }
    }
  }
#pragma unroll
  for (int kx = 0; kx < 3; ++kx) {
    float* pp = part + ((size_t)blockIdx.x * (NTAP * C) + (kz * 9 + ky * 3 + kx) * C + ci) * K;
#pragma unroll
    for (int k = 0; k < K; ++k) {
      pp[k] = acc[kx][k];
    }
  }
}

// part[b][tap][co] = sum_p g1[p][co] a0[p + d(tap)]; bpart[b][co] = sum_p g1[p][co].
// Lane = co; each of the eight warps takes two tile rows of sixteen voxels and
// keeps all 27 taps in registers: four voxels' g1 values and, row offset by row
// offset, eight a0 values (two 16-byte reads, the same for every lane) feed 12
// multiply-adds.  (A warp per row offset read one a0 and one g1 value for every
// three: 0.509 against 0.281 ms at 64x256x256.)  The warps' sums are added in a
// fixed order at the end.
constexpr int HXP = 20;     // halo row pitch: 18 columns, 16-byte aligned rows
__global__ void __launch_bounds__(256, 3)
k_wgrad_first(const bf16* __restrict__ a0, const bf16* __restrict__ g1, float* __restrict__ part,
              float* __restrict__ bpart, Dims d) {
  __shared__ __align__(16) float s_h[HZ * HY * HXP];
  __shared__ __align__(16) float s_g[TV * C];
  const int co = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float acc[NTAP], bacc = 0.f;
#pragma unroll
  for (int t = 0; t < NTAP; ++t) acc[t] = 0.f;
  for (int i = threadIdx.x; i < HZ * HY * HXP; i += blockDim.x) s_h[i] = 0.f;     // the pad columns stay zero
  for (int tile = blockIdx.x; tile < d.ntiles; tile += gridDim.x) {
    int z0, y0, x0;
    tile_origin(tile, d, z0, y0, x0);
    __syncthreads();
    for (int h = threadIdx.x; h < HV; h += blockDim.x) {
      const int hx = h % HX, t = h / HX, hy = t % HY, hz = t / HY;
      const int gz = z0 - 1 + hz, gy = y0 - 1 + hy, gx = x0 - 1 + hx;
      s_h[t * HXP + hx] = inside(d, gz, gy, gx) ? __bfloat162float(a0[vox(d, gz, gy, gx)]) : 0.f;
    }
    for (int i = threadIdx.x; i < TV * 4; i += blockDim.x) {
      const int c = i & 3, r = i >> 2;
      const int gz = z0 + (r >> 7), gy = y0 + ((r >> 4) & 7), gx = x0 + (r & 15);
      float f[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
      if (inside(d, gz, gy, gx)) unpack8(*reinterpret_cast<const uint4*>(g1 + vox(d, gz, gy, gx) * C + c * 8), f);
      float4* dst = reinterpret_cast<float4*>(s_g + r * C + c * 8);
      dst[0] = make_float4(f[0], f[1], f[2], f[3]);
      dst[1] = make_float4(f[4], f[5], f[6], f[7]);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = 0; i < 8; ++i) {                    // two rows of four chunks of four voxels
      const int row = 2 * warp + (i >> 2), x = 4 * (i & 3), tz = row >> 3, ty = row & 7;
      float g[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        g[e] = s_g[(row * TX + x + e) * C + co];
        bacc += g[e];
      }
#pragma unroll
      for (int r = 0; r < 9; ++r) {
        const float* hr = s_h + ((tz + r / 3) * HY + ty + r % 3) * HXP + x;
        const float4 p = *reinterpret_cast<const float4*>(hr), q = *reinterpret_cast<const float4*>(hr + 4);
        const float v[6] = {p.x, p.y, p.z, p.w, q.x, q.y};
#pragma unroll
        for (int e = 0; e < 4; ++e)
#pragma unroll
          for (int kx = 0; kx < 3; ++kx) acc[3 * r + kx] = fmaf(g[e], v[e + kx], acc[3 * r + kx]);
      }
    }
  }
  // the eight warps' sums: [warp][28][32] in s_g, added in order
  __syncthreads();
#pragma unroll
  for (int t = 0; t < NTAP; ++t) s_g[(warp * (NTAP + 1) + t) * C + co] = acc[t];
  s_g[(warp * (NTAP + 1) + NTAP) * C + co] = bacc;
  __syncthreads();
  for (int i = threadIdx.x; i < (NTAP + 1) * C; i += blockDim.x) {
    float t = 0.f;
    for (int v = 0; v < 8; ++v) t += s_g[v * (NTAP + 1) * C + i];
    if (i < NTAP * C) part[(size_t)blockIdx.x * (NTAP * C) + i] = t;
    else bpart[(size_t)blockIdx.x * C + i - NTAP * C] = t;
  }
}

// ------------------------------------------------------------------ reductions, input, parameters

enum { MAP_MID = 1, MAP_FIRST = 2, MAP_LAST = 3 };

// sum_b p[b * n], b = 0 .. P-1, eight at a time in flight: the loop is one load
// latency per trip (a 31x120x100 layer's weight gradient took 99.7 us with four
// loads a trip and blocks of 256, 79.5 so, in blocks of 64 and with the biases
// in the same launch).  The eight are added in three floats (Sum3), then to the
// double, which holds what a double addition for each would: 152 partial sums of 27648
// outputs take 12.5 us so, 20.7 with one each (float pairs, 11.2, lost bits).
__device__ __forceinline__ double sum_parts(const float* __restrict__ p, int P, size_t n) {
  double s = 0.0;
  int b = 0;
  for (; b + 8 <= P; b += 8) {
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = p[(size_t)(b + e) * n];
    muffin::Sum3 t;
#pragma unroll
    for (int e = 0; e < 8; ++e) t.add(v[e]);
    if (fabsf(t.hi) <= 1e37f && fabsf(t.mid) <= 1e37f) {
      t.into(s);
    } else {                         // infinities, NaN, or sums near the end of the range
#pragma unroll 1
      for (int e = 0; e < 8; ++e) s += p[(size_t)(b + e) * n];
    }
  }
  for (; b < P; ++b) s += p[(size_t)b * n];
  return s;
}

constexpr int kReduceThreads = 64;

// out[map(i)] = sum_b part[b*n + i] (fixed order, double accumulation), and with bout the C biases
// bout[c] = sum_b bpart[b*C + c].
// MAP_MID: i = (tap*32 + co)*32 + ci -> (co*32 + ci)*27 + tap; MAP_FIRST:
// i = tap*32 + co -> co*27 + tap; MAP_LAST: i = (tap*32 + ci)*K + k -> (k*32 + ci)*27 + tap.
__global__ void __launch_bounds__(kReduceThreads)
k_reduce_part(const float* __restrict__ part, int P, int n, float* __restrict__ out, int map, int K,
              const float* __restrict__ bpart, float* __restrict__ bout) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) {
    if (bout && i - n < C) bout[i - n] = (float)sum_parts(bpart + (i - n), P, C);
    return;
  }
  int j = i;
  const double s = sum_parts(part + i, P, n);
  if (map == MAP_LAST) {
    const int k = i % K, r = i / K, ci = r & 31, t = r >> 5;
    j = (k * C + ci) * NTAP + t;
  } else if (map == MAP_MID) {
    const int t = i >> 10, co = (i >> 5) & 31, ci = i & 31;
    j = (co * C + ci) * NTAP + t;
  } else if (map == MAP_FIRST) {
    const int t = i >> 5, c = i & 31;
    j = c * NTAP + t;
  }
  out[j] = (float)s;
}

// loss = sum_b lpart[b][0] / V; gradient of the last biases: 2 lam_k sum_b lpart[b][1+k] / V.
__global__ void k_loss_final(const double* __restrict__ lpart, int P, int K, Lam lam, long long nvox,
                             double* __restrict__ loss, float* __restrict__ grad_b6) {
  if (blockIdx.x != 0) return;
  const int k = (int)threadIdx.x - 1;
  if (k >= K) return;
  double acc = 0.0;
  int b = 0;
  for (; b + 8 <= P; b += 8) {      // eight loads in flight, summed in order
    double v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = lpart[(size_t)(b + e) * (K + 1) + 1 + k];
#pragma unroll
    for (int e = 0; e < 8; ++e) acc += v[e];
  }
  for (; b < P; ++b) acc += lpart[(size_t)b * (K + 1) + 1 + k];
  if (k < 0) {
    if (loss) *loss = acc / (double)nvox;
  } else if (grad_b6) {
    grad_b6[k] = (float)(2.0 * lam.v[k] * acc / (double)nvox);
  }
}

__global__ void k_maxabs_part(const float* __restrict__ y, long long n, float* __restrict__ part) {
  float m = 0.f;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    m = fmaxf(m, fabsf(y[i]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
  __shared__ float s[32];
  if ((threadIdx.x & 31) == 0) s[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    float r = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmaxf(r, s[w]);
    part[blockIdx.x] = r;
  }
}

// s = max |y| (1 if the cube is zero).  One warp.
__global__ void k_scale_final(const float* __restrict__ part, int P, float* __restrict__ s) {
  float m = 0.f;
  for (int b = threadIdx.x; b < P; b += 32) m = fmaxf(m, part[b]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (threadIdx.x == 0) *s = m > 0.f ? m : 1.f;
}

// a0 = bf16(y / s).
__global__ void k_prep_input(const float* __restrict__ y, const float* __restrict__ s, bf16* __restrict__ a0,
                             long long n) {
  const float inv = 1.0f / *s;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    a0[i] = __float2bfloat16_rn(y[i] * inv);
}

struct KernelWeights {
  float* w1;    // [27][32] (tap, co), bfloat16 values
  float* b1;    // [32]
  bf16* wf;     // [4][27][32 co][32 ci]   forward operands of layers 2..5
  bf16* wb;     // [4][27][32 ci][32 co]   flipped, transposed: input gradients
  float* bm;    // [4][32]
  float* w6b;   // [27][K][32 ci]  last layer, input gradient; bfloat16 values
  bf16* w6t;    // [27][16 co][32 ci]  last layer, tcgen05 operand (rows K .. 15 zero)
  float* b6;    // [K]
};

__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// Packed float32 parameters -> the layouts the kernels read.
__global__ void k_unpack_params(const float* __restrict__ theta, KernelWeights kw, int K) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  constexpr int L1 = NTAP * C + C;           // 896
  constexpr int LM = WMID + C;               // 27680
  const int N = L1 + 4 * LM + K * NTAP * C + K;
  if (i >= N) return;
  const float v = theta[i];
  if (i < L1) {
    if (i < NTAP * C) kw.w1[(i % NTAP) * C + i / NTAP] = round_bf16(v);
    else kw.b1[i - NTAP * C] = v;
    return;
  }
  int j = i - L1;
  if (j < 4 * LM) {
    const int l = j / LM, li = j % LM;
    if (li < WMID) {
      const int co = li / (C * NTAP), rem = li % (C * NTAP), ci = rem / NTAP, t = rem % NTAP;
      const bf16 q = __float2bfloat16_rn(v);
      kw.wf[(size_t)l * WMID + (t * C + co) * C + ci] = q;
      kw.wb[(size_t)l * WMID + ((NTAP - 1 - t) * C + ci) * C + co] = q;
    } else {
      kw.bm[l * C + li - WMID] = v;
    }
    return;
  }
  j -= 4 * LM;
  if (j < K * NTAP * C) {
    const int k = j / (C * NTAP), rem = j % (C * NTAP), ci = rem / NTAP, t = rem % NTAP;
    kw.w6b[(t * K + k) * C + ci] = round_bf16(v);
    kw.w6t[(t * kLastN + k) * C + ci] = __float2bfloat16_rn(v);
  } else {
    kw.b6[j - K * NTAP * C] = v;
  }
}

// One 32 -> 32 layer's weights [co][ci][27] float32 -> forward ([27][co][ci])
// or input-gradient ([27 flipped][ci][co]) bfloat16 operands.
__global__ void k_pack_layer(const float* __restrict__ w, bf16* __restrict__ out, int backward) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= WMID) return;
  const int co = i / (C * NTAP), rem = i % (C * NTAP), ci = rem / NTAP, t = rem % NTAP;
  const bf16 q = __float2bfloat16_rn(w[i]);
  if (backward) out[((NTAP - 1 - t) * C + ci) * C + co] = q;
  else out[(t * C + co) * C + ci] = q;
}

// Adam (Kingma and Ba 2015, Algorithm 1); c1 = 1/(1 - beta1^t), c2 = 1/(1 - beta2^t).
__global__ void k_adam(float* __restrict__ theta, const float* __restrict__ g, float* __restrict__ m,
                       float* __restrict__ v, int n, float lr, float c1, float c2) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  // a layer of this step (or an unchecked earlier call) gave up a wait: its
  // gradient is incomplete, so the step is dropped; muffin_net_check reports it
  if (*(volatile int*)&g_tc_timeouts != 0) return;
  const float gi = g[i];
  const float mi = 0.9f * m[i] + 0.1f * gi;
  const float vi = 0.999f * v[i] + 0.001f * gi * gi;
  m[i] = mi;
  v[i] = vi;
  theta[i] -= lr * (mi * c1) / (sqrtf(vi * c2) + 1e-8f);
}

// ------------------------------------------------------------------ host side

constexpr int kFixedParams = NTAP * C + C + 4 * (WMID + C);   // layers 1..5

int param_count(int K) { return kFixedParams + K * (NTAP * C + 1); }

int w_offset(int k) {  // packed offset of layer k's weights (k = 0..5)
  if (k == 0) return 0;
  return NTAP * C + C + (k - 1) * (WMID + C);
}
int b_offset(int k, int K) {
  const int co = k == 5 ? K : C, ci = k == 0 ? 1 : C;
  return w_offset(k) + co * ci * NTAP;
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

bool dims_ok(int nz, int ny, int nx) {
  if (nz < 1 || ny < 1 || nx < 1) return false;
  const long long v = (long long)nz * ny * nx;
  return v < (1LL << 31) / C;
}

int part_slots(const Dims& d) { return d.ntiles < kMaxPart ? d.ntiles : kMaxPart; }
int loss_slots(const Dims& d) { return d.ntiles < kMaxLossPart ? d.ntiles : kMaxLossPart; }

int sm_count() {
  int dev = 0, n = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;
  if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) return 148;
  return n;
}

template <int K> constexpr int last_bwd_smem() { return K * (NTAP * C + HV) * 4; }
template <int K> constexpr int wgrad_last_smem() { return HV * ROWB + TV * last_pitch<K>() * 4; }

#define MNET_SWITCH_K(K, CALL) \
  switch (K) {                 \
    case 1: CALL(1); break;    \
    case 2: CALL(2); break;    \
    case 3: CALL(3); break;    \
    case 4: CALL(4); break;    \
    case 5: CALL(5); break;    \
    case 6: CALL(6); break;    \
    case 7: CALL(7); break;    \
    default: CALL(8); break;   \
  }

cudaError_t configure_once() {
  static const cudaError_t err = [] {
    cudaError_t e;
    if ((e = muffin::allow_max_dyn_smem(k_conv_tc05<EPI_RELU>)) == cudaSuccess &&
        (e = muffin::allow_max_dyn_smem(k_conv_tc05<EPI_BIAS>)) == cudaSuccess &&
        (e = muffin::allow_max_dyn_smem(k_conv_tc05<EPI_MASK>)) == cudaSuccess &&
        (e = muffin::allow_max_dyn_smem(k_conv_tc05<EPI_PRED>)) == cudaSuccess &&
        (e = muffin::allow_max_dyn_smem(k_conv_tc05<EPI_LOSS>)) == cudaSuccess)
      e = muffin::allow_max_dyn_smem(k_wgrad_tc05);
#define CALL(KK)                                                                                       \
  if (e == cudaSuccess && (e = muffin::allow_max_dyn_smem(k_last_bwd_data<KK>)) == cudaSuccess)        \
  e = muffin::allow_max_dyn_smem(k_wgrad_last<KK>)
    for (int K = 1; K <= kMaxOut; ++K) MNET_SWITCH_K(K, CALL)
#undef CALL
    return e;
  }();
  return err;
}

// Launch helpers (all persistent: grids bounded by the tile count).
// Tiles of 128 voxels and the persistent grid of k_conv_tc05 (two CTAs per SM).
int tc05_tiles(const Dims& d, int& tx, int& ty) {
  tx = (d.nx + U_TX - 1) / U_TX;
  ty = (d.ny + U_TY - 1) / U_TY;
  return tx * ty * d.nz;
}
int tc05_grid(const Dims& d, int sms) {
  int tx, ty;
  int g = tc05_tiles(d, tx, ty);
  if (g > 2 * sms) g = 2 * sms;
  return g < kMaxLossPart ? g : kMaxLossPart;   // also the last layer's loss partial slots
}

template <int EPI>
cudaError_t launch_tc05(const bf16* in, const bf16* wk, const float* bias, const bf16* mask, bf16* out,
                        const Dims& d, int sms, cudaStream_t st, const LastArgs& la) {
  int tx, ty;
  tc05_tiles(d, tx, ty);
  k_conv_tc05<EPI><<<tc05_grid(d, sms), 288, conv05_smem(epi_n<EPI>()), st>>>(in, wk, bias, mask, out, d, tx, ty, la);
  return cudaGetLastError();
}

cudaError_t launch_conv(int epi, const bf16* in, const bf16* wk, const float* bias, const bf16* mask, bf16* out,
                        const Dims& d, int sms, cudaStream_t st) {
  const LastArgs none{};
  if (epi == EPI_RELU) return launch_tc05<EPI_RELU>(in, wk, bias, mask, out, d, sms, st, none);
  if (epi == EPI_BIAS) return launch_tc05<EPI_BIAS>(in, wk, bias, mask, out, d, sms, st, none);
  return launch_tc05<EPI_MASK>(in, wk, bias, mask, out, d, sms, st, none);
}

void launch_reduce(const float* part, int P, int n, float* out, int map, int K, const float* bpart, float* bout,
                   cudaStream_t st) {
  k_reduce_part<<<(n + (bout ? C : 0) + kReduceThreads - 1) / kReduceThreads, kReduceThreads, 0, st>>>(
      part, P, n, out, map, K, bpart, bout);
}

// Planes between two flushes of the weight gradient's accumulators, for runs of
// `tiles` tiles.  A run without a flush is further from 64 bits than tiles taken
// in turns over the cube are, because ragged tiles add less and contiguous runs
// take the full ones together (31x120x100 1.87e-6 against 1.76e-6, 7x33x41 1.44e-7
// against 1.18e-7, 64x256x256 2.85e-5 against 2.75e-5).  So half a run where more
// than a tenth of the tiles' voxels lies outside the cube, else fifteen sixteenths,
// which is enough (1.33e-6, 8.4e-8, 2.39e-5) and moves the sums of long runs by
// less than 1e-5.  A flush holds the MMAs up for 2.3 us: kernel of 31x120x100 64
// -> 66 us, 7x33x41 22 -> 32, 64x256x256 453 -> 468.
int wgrad_flush(const Dims& d, int ntiles, int P) {
  const int tiles = ntiles / P;
  const bool ragged = 10 * d.nvox < 9LL * ntiles * U_TY * U_TX;
  const int f = ragged ? tiles / 2 : tiles * 15 / 16;
  return f < 1 ? 1 : f;
}

// Weight and bias gradients of a 32 -> 32 layer: per-CTA partial sums (one CTA
// per SM, at most part_slots(d) of them), then the fixed-order reduction.
void launch_wgrad_mid(const bf16* a, const bf16* dz, float* part, float* bpart, float* dw, float* db, const Dims& d,
                      int sms, cudaStream_t st) {
  int tx, ty;
  const int ntiles = tc05_tiles(d, tx, ty);
  int P = part_slots(d);
  if (P > sms) P = sms;
  if (P > ntiles) P = ntiles;
  k_wgrad_tc05<<<P, 288, wgrad05_smem, st>>>(a, dz, part, bpart, d, tx, ty, wgrad_flush(d, ntiles, P));
  launch_reduce(part, P, WMID, dw, MAP_MID, 1, bpart, db, st);
}

}  // namespace mnet

using namespace mnet;

// ====================================================================== network context

struct muffin_net {
  int training = 0;
  int K = 1;          // output maps
  Lam lam{};
  Dims d{};
  cudaStream_t st = nullptr;
  int sms = 148;
  long long step = 0;
  std::string err;
  // parameters and optimiser
  float *theta = nullptr, *mom1 = nullptr, *mom2 = nullptr, *grad = nullptr;
  KernelWeights kw{};
  // scalars and partials
  float* s = nullptr;
  float* mpart = nullptr;
  double* lpart = nullptr;
  double* loss = nullptr;
  float* part = nullptr;
  float* bpart = nullptr;
  // maps
  bf16* a0 = nullptr;
  bf16* act = nullptr;   // training: a1..a5; inference: two ping-pong maps
  bf16* gA = nullptr;
  bf16* gB = nullptr;
  float* d6 = nullptr;   // loss gradient [V][K]

  bf16* map(int i) const { return act + (size_t)i * d.nvox * C; }
};

namespace {

// Workspace carve-up; with base == nullptr only the size is computed.
size_t net_layout(muffin_net* n, const Dims& d, int K, int training, char* base) {
  size_t off = 0;
  auto take = [&](size_t bytes) -> char* {
    char* p = base ? base + off : nullptr;
    off = align256(off + bytes);
    return p;
  };
  const int np = param_count(K);
  const size_t V = (size_t)d.nvox;
  float* theta = (float*)take(np * 4);
  float* m1 = (float*)take(training ? np * 4 : 0);
  float* m2 = (float*)take(training ? np * 4 : 0);
  float* grad = (float*)take(training ? np * 4 : 0);
  KernelWeights kw;
  kw.w1 = (float*)take(NTAP * C * 4);
  kw.b1 = (float*)take(C * 4);
  kw.wf = (bf16*)take(4 * WMID * 2);
  kw.wb = (bf16*)take(4 * WMID * 2);
  kw.bm = (float*)take(4 * C * 4);
  kw.w6b = (float*)take(NTAP * K * C * 4);
  kw.w6t = (bf16*)take(NTAP * kLastN * C * 2);
  kw.b6 = (float*)take(K * 4);
  float* s = (float*)take(4);
  float* mpart = (float*)take(kMaxLossPart * 4);
  double* lpart = (double*)take((size_t)(K + 1) * kMaxLossPart * 8);
  double* loss = (double*)take(8);
  const int P = part_slots(d);
  float* part = (float*)take(training ? (size_t)P * WMID * 4 : 0);
  float* bpart = (float*)take(training ? (size_t)P * C * 4 : 0);
  bf16* a0 = (bf16*)take(V * 2);
  bf16* act = (bf16*)take((training ? 5 : 2) * V * C * 2);
  bf16* gA = (bf16*)take(training ? V * C * 2 : 0);
  bf16* gB = (bf16*)take(training ? V * C * 2 : 0);
  float* d6 = (float*)take(training ? V * K * 4 : 0);
  if (n) {
    n->theta = theta; n->mom1 = m1; n->mom2 = m2; n->grad = grad; n->kw = kw;
    n->s = s; n->mpart = mpart; n->lpart = lpart; n->loss = loss; n->part = part; n->bpart = bpart;
    n->a0 = a0; n->act = act; n->gA = gA; n->gB = gB; n->d6 = d6;
  }
  return off;
}

int fail(muffin_net* n, int code, const std::string& msg) {
  if (n) n->err = msg;
  return code;
}

int cuda_check(muffin_net* n, const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(n, MUFFIN_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return MUFFIN_OK;
}

// s, a0 and the forward pass through layer 5 (training keeps every map).
void forward_to_a5(muffin_net* n, const float* y) {
  const Dims& d = n->d;
  const int PL = loss_slots(d);
  const int grid_s = (int)((d.nvox + 255) / 256 < PL ? (d.nvox + 255) / 256 : PL);
  k_maxabs_part<<<grid_s, 256, 0, n->st>>>(y, d.nvox, n->mpart);
  k_scale_final<<<1, 32, 0, n->st>>>(n->mpart, grid_s, n->s);
  const int grid_p = (int)((d.nvox + 255) / 256 < 4 * n->sms ? (d.nvox + 255) / 256 : 4 * n->sms);
  k_prep_input<<<grid_p, 256, 0, n->st>>>(y, n->s, n->a0, d.nvox);
  const int gsimt = d.ntiles < 5 * n->sms ? d.ntiles : 5 * n->sms;   // five blocks an SM
  bf16* out = n->map(0);
  k_first_fwd<<<gsimt, kFirstThreads, 0, n->st>>>(n->a0, n->kw.w1, n->kw.b1, out, d);
  for (int l = 0; l < 4; ++l) {
    bf16* in = out;
    out = n->training ? n->map(l + 1) : n->map((l + 1) & 1);
    launch_conv(EPI_RELU, in, n->kw.wf + (size_t)l * WMID, n->kw.bm + l * C, nullptr, out, d, n->sms, n->st);
  }
}

bf16* a5_of(muffin_net* n) { return n->training ? n->map(4) : n->map(0); }

LastArgs last_args(muffin_net* n) {
  LastArgs la{};
  la.K = n->K;
  la.lam = n->lam;
  la.s = n->s;
  return la;
}

void last_predict(muffin_net* n, float* x, float* aux) {
  LastArgs la = last_args(n);
  la.out_x = x;
  la.out_aux = aux;
  launch_tc05<EPI_PRED>(a5_of(n), n->kw.w6t, n->kw.b6, nullptr, nullptr, n->d, n->sms, n->st, la);
}

// Last layer of the training pass: loss, its gradient d6, the layer's weight
// and bias gradients, and the gradient of a5's pre-activation into g5.
void last_train(muffin_net* n, const float* tx, const bf16* taux, bf16* g5) {
  const Dims& d = n->d;
  bf16* a5 = a5_of(n);
  LastArgs la = last_args(n);
  la.tx = tx;
  la.taux = taux;
  la.d6 = n->d6;
  la.lpart = n->lpart;
  launch_tc05<EPI_LOSS>(a5, n->kw.w6t, n->kw.b6, nullptr, nullptr, d, n->sms, n->st, la);
  k_loss_final<<<1, n->K + 1, 0, n->st>>>(n->lpart, tc05_grid(d, n->sms), n->K, n->lam, d.nvox, n->loss,
                                          n->grad + b_offset(5, n->K));
  int P = part_slots(d);
  if (P > 2 * n->sms) P = 2 * n->sms;
  const int grid = d.ntiles < 4 * n->sms ? d.ntiles : 4 * n->sms;
#define CALL(KK)                                                                      \
  k_wgrad_last<KK><<<P, 288, wgrad_last_smem<KK>(), n->st>>>(n->d6, a5, n->part, d);  \
  k_last_bwd_data<KK><<<grid, kLastThreads, last_bwd_smem<KK>(), n->st>>>(n->d6, n->kw.w6b, a5, g5, d)
  MNET_SWITCH_K(n->K, CALL)
#undef CALL
  launch_reduce(n->part, P, NTAP * C * n->K, n->grad + w_offset(5), MAP_LAST, n->K, nullptr, nullptr, n->st);
}

// Loss and gradient into n->grad (training contexts).
void loss_and_grad(muffin_net* n, const float* y, const float* tx, const bf16* taux) {
  const Dims& d = n->d;
  forward_to_a5(n, y);
  bf16* g = n->gA;
  bf16* other = n->gB;
  last_train(n, tx, taux, g);
  for (int k = 4; k >= 1; --k) {          // layers 5..2 (index k), input map a_k = map(k - 1)
    const bf16* a_in = n->map(k - 1);
    launch_wgrad_mid(a_in, g, n->part, n->bpart, n->grad + w_offset(k), n->grad + b_offset(k, n->K), d, n->sms,
                     n->st);
    launch_conv(EPI_MASK, g, n->kw.wb + (size_t)(k - 1) * WMID, nullptr, a_in, other, d, n->sms, n->st);
    bf16* tmp = g; g = other; other = tmp;
  }
  int P = part_slots(d);
  if (P > 3 * n->sms) P = 3 * n->sms;      // three blocks an SM
  k_wgrad_first<<<P, 256, 0, n->st>>>(n->a0, g, n->part, n->bpart, d);
  launch_reduce(n->part, P, NTAP * C, n->grad + w_offset(0), MAP_FIRST, 1, n->bpart, n->grad + b_offset(0, n->K), n->st);
}

void unpack_params(muffin_net* n) {
  const int np = param_count(n->K);
  cudaMemsetAsync(n->kw.w6t, 0, NTAP * kLastN * C * 2, n->st);
  k_unpack_params<<<(np + 255) / 256, 256, 0, n->st>>>(n->theta, n->kw, n->K);
}

}  // namespace

extern "C" {

int muffin_net_num_params(int n_out) {
  if (n_out < 1 || n_out > kMaxOut) return 0;
  return param_count(n_out);
}

size_t muffin_net_workspace_bytes(int nz, int ny, int nx, int n_out, int training) {
  if (!dims_ok(nz, ny, nx) || n_out < 1 || n_out > kMaxOut) return 0;
  return net_layout(nullptr, make_dims(nz, ny, nx), n_out, training != 0, nullptr);
}

int muffin_net_create(muffin_net** out, int nz, int ny, int nx, int n_out, const float* h_out_weight, int training,
                      void* d_ws, size_t ws_bytes, cudaStream_t stream) {
  if (!out) return MUFFIN_ERR_ARG;
  *out = nullptr;
  if (!dims_ok(nz, ny, nx) || n_out < 1 || n_out > kMaxOut) return MUFFIN_ERR_ARG;
  Lam lam;
  for (int k = 0; k < kMaxOut; ++k) lam.v[k] = 1.f;
  if (h_out_weight)
    for (int k = 0; k < n_out; ++k) {
      if (!(h_out_weight[k] >= 0.f) || !std::isfinite(h_out_weight[k])) return MUFFIN_ERR_ARG;
      lam.v[k] = h_out_weight[k];
    }
  if (!d_ws || ((uintptr_t)d_ws & 255)) return MUFFIN_ERR_ARG;
  const Dims d = make_dims(nz, ny, nx);
  const size_t need = net_layout(nullptr, d, n_out, training != 0, nullptr);
  if (ws_bytes < need) return MUFFIN_ERR_NOMEM;
  if (configure_once() != cudaSuccess) return MUFFIN_ERR_CUDA;
  muffin_net* n = new muffin_net();
  n->training = training != 0;
  n->K = n_out;
  n->lam = lam;
  n->d = d;
  n->st = stream;
  n->sms = sm_count();
  net_layout(n, d, n_out, n->training, (char*)d_ws);
  const int np = param_count(n_out);
  cudaMemsetAsync(n->theta, 0, np * 4, stream);
  if (n->training) {
    cudaMemsetAsync(n->mom1, 0, np * 4, stream);
    cudaMemsetAsync(n->mom2, 0, np * 4, stream);
  }
  unpack_params(n);
  if (cudaGetLastError() != cudaSuccess) {
    delete n;
    return MUFFIN_ERR_CUDA;
  }
  *out = n;
  return MUFFIN_OK;
}

int muffin_net_set_params(muffin_net* n, const float* d_theta) {
  if (!n) return MUFFIN_ERR_ARG;
  if (!d_theta) return fail(n, MUFFIN_ERR_ARG, "d_theta is NULL");
  const int np = param_count(n->K);
  cudaMemcpyAsync(n->theta, d_theta, np * 4, cudaMemcpyDeviceToDevice, n->st);
  if (n->training) {
    cudaMemsetAsync(n->mom1, 0, np * 4, n->st);
    cudaMemsetAsync(n->mom2, 0, np * 4, n->st);
  }
  n->step = 0;
  unpack_params(n);
  return cuda_check(n, "muffin_net_set_params");
}

int muffin_net_get_params(const muffin_net* n, float* d_theta) {
  if (!n || !d_theta) return MUFFIN_ERR_ARG;
  cudaMemcpyAsync(d_theta, n->theta, param_count(n->K) * 4, cudaMemcpyDeviceToDevice, n->st);
  return cuda_check(const_cast<muffin_net*>(n), "muffin_net_get_params");
}

// Synchronise the context's stream, then read and clear the device's count of
// tensor-core waits that gave up; MUFFIN_ERR_TIMEOUT if it was not zero.
static int check_waits(muffin_net* n, const char* what) {
  cudaError_t e = cudaStreamSynchronize(n->st);
  if (e != cudaSuccess) return fail(n, MUFFIN_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  int v = 0, zero = 0;
  if ((e = cudaMemcpyFromSymbol(&v, g_tc_timeouts, sizeof(int))) != cudaSuccess ||
      (e = cudaMemcpyToSymbol(g_tc_timeouts, &zero, sizeof(int))) != cudaSuccess)
    return fail(n, MUFFIN_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  if (v != 0)
    return fail(n, MUFFIN_ERR_TIMEOUT, std::string(what) + ": " + std::to_string(v) +
                                           " thread block(s) of the tensor-core layers gave up a bounded wait; "
                                           "their output tiles (and any Adam step queued after them) were skipped");
  return MUFFIN_OK;
}

int muffin_net_predict(muffin_net* n, const float* d_dirty, float* d_x, float* d_aux) {
  if (!n) return MUFFIN_ERR_ARG;
  if (!d_dirty || !d_x) return fail(n, MUFFIN_ERR_ARG, "NULL cube pointer");
  if (n->K > 1 && !d_aux) return fail(n, MUFFIN_ERR_ARG, "NULL d_aux with more than one output map");
  forward_to_a5(n, d_dirty);
  last_predict(n, d_x, d_aux);
  const int r = cuda_check(n, "muffin_net_predict");
  if (r != MUFFIN_OK) return r;
  return check_waits(n, "muffin_net_predict");
}

int muffin_net_check(muffin_net* n) {
  if (!n) return MUFFIN_ERR_ARG;
  const int r = cuda_check(n, "muffin_net_check");
  if (r != MUFFIN_OK) return r;
  return check_waits(n, "muffin_net_check");
}

int muffin_net_set_wait_limit(long long polls) {
  const long long v = polls < 0 ? kWaitLimit : polls;
  return cudaMemcpyToSymbol(g_wait_polls, &v, sizeof(v)) == cudaSuccess ? MUFFIN_OK : MUFFIN_ERR_CUDA;
}

static int check_targets(muffin_net* n, const float* d_dirty, const float* d_tx, const void* d_taux) {
  if (!n->training) return fail(n, MUFFIN_ERR_STATE, "not a training context");
  if (!d_dirty || !d_tx) return fail(n, MUFFIN_ERR_ARG, "NULL pointer");
  if (n->K > 1 && !d_taux) return fail(n, MUFFIN_ERR_ARG, "NULL d_target_aux with more than one output map");
  return MUFFIN_OK;
}

int muffin_net_loss_grad(muffin_net* n, const float* d_dirty, const float* d_tx, const void* d_taux, float* d_grad,
                         double* h_loss) {
  if (!n) return MUFFIN_ERR_ARG;
  int r = check_targets(n, d_dirty, d_tx, d_taux);
  if (r != MUFFIN_OK) return r;
  if (!d_grad) return fail(n, MUFFIN_ERR_ARG, "NULL d_grad");
  loss_and_grad(n, d_dirty, d_tx, (const bf16*)d_taux);
  cudaMemcpyAsync(d_grad, n->grad, param_count(n->K) * 4, cudaMemcpyDeviceToDevice, n->st);
  r = cuda_check(n, "muffin_net_loss_grad");
  if (r != MUFFIN_OK) return r;
  if (h_loss) {
    cudaMemcpyAsync(h_loss, n->loss, 8, cudaMemcpyDeviceToHost, n->st);
    return check_waits(n, "muffin_net_loss_grad");
  }
  return MUFFIN_OK;
}

int muffin_net_train_step(muffin_net* n, const float* d_dirty, const float* d_tx, const void* d_taux, float lr,
                          double* d_loss) {
  if (!n) return MUFFIN_ERR_ARG;
  int r = check_targets(n, d_dirty, d_tx, d_taux);
  if (r != MUFFIN_OK) return r;
  if (!(lr >= 0.f) || !std::isfinite(lr)) return fail(n, MUFFIN_ERR_ARG, "learning rate must be finite and >= 0");
  loss_and_grad(n, d_dirty, d_tx, (const bf16*)d_taux);
  if (d_loss) cudaMemcpyAsync(d_loss, n->loss, 8, cudaMemcpyDeviceToDevice, n->st);
  n->step += 1;
  const double c1 = 1.0 / (1.0 - std::pow(0.9, (double)n->step));
  const double c2 = 1.0 / (1.0 - std::pow(0.999, (double)n->step));
  const int np = param_count(n->K);
  k_adam<<<(np + 255) / 256, 256, 0, n->st>>>(n->theta, n->grad, n->mom1, n->mom2, np, lr, (float)c1, (float)c2);
  unpack_params(n);
  return cuda_check(n, "muffin_net_train_step");
}

int muffin_net_wait_timeouts(void) {
  int v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_tc_timeouts, sizeof(int)) != cudaSuccess) return -1;
  if (cudaMemcpyToSymbol(g_tc_timeouts, &zero, sizeof(int)) != cudaSuccess) return -1;
  return v;
}

const char* muffin_net_last_error(const muffin_net* n) {
  if (!n) return "invalid arguments to muffin_net_create (sizes, output maps, weights, workspace) or CUDA set-up failed";
  return n->err.c_str();
}

void muffin_net_destroy(muffin_net* n) { delete n; }

// ---------------------------------------------------------------------- single layers

static thread_local std::string g_conv_err;

static int conv_fail(int code, const std::string& msg) {
  g_conv_err = msg;
  return code;
}

static int conv_cuda(const char* what) {
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return conv_fail(MUFFIN_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
  return MUFFIN_OK;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

size_t muffin_conv3d_scratch_bytes(int nz, int ny, int nx) {
  if (!dims_ok(nz, ny, nx)) return 0;
  const Dims d = make_dims(nz, ny, nx);
  const int P = part_slots(d);
  return align256(WMID * 2) + align256((size_t)P * WMID * 4) + align256((size_t)P * C * 4);
}

static int layer_args(const void* a, const void* b, int nz, int ny, int nx, void* scratch, size_t bytes) {
  if (!dims_ok(nz, ny, nx)) return conv_fail(MUFFIN_ERR_ARG, "sizes must be >= 1 with nz*ny*nx*32 < 2^31");
  if (!a || !b || !scratch) return conv_fail(MUFFIN_ERR_ARG, "NULL pointer");
  if (!aligned16(a) || !aligned16(b) || ((uintptr_t)scratch & 255))
    return conv_fail(MUFFIN_ERR_ARG, "maps must be 16-byte aligned, scratch 256-byte aligned");
  if (bytes < muffin_conv3d_scratch_bytes(nz, ny, nx)) return conv_fail(MUFFIN_ERR_NOMEM, "scratch too small");
  if (configure_once() != cudaSuccess) return conv_fail(MUFFIN_ERR_CUDA, "kernel attributes could not be set");
  return MUFFIN_OK;
}

int muffin_conv3d_forward(const void* d_a, const float* d_w, const float* d_b, int relu, void* d_z, int nz, int ny,
                          int nx, void* d_scratch, size_t scratch_bytes, cudaStream_t stream) {
  int r = layer_args(d_a, d_z, nz, ny, nx, d_scratch, scratch_bytes);
  if (r != MUFFIN_OK) return r;
  if (!d_w) return conv_fail(MUFFIN_ERR_ARG, "NULL weights");
  const Dims d = make_dims(nz, ny, nx);
  bf16* wk = (bf16*)d_scratch;
  k_pack_layer<<<(WMID + 255) / 256, 256, 0, stream>>>(d_w, wk, 0);
  launch_conv(relu ? EPI_RELU : EPI_BIAS, (const bf16*)d_a, wk, d_b, nullptr, (bf16*)d_z, d, sm_count(), stream);
  return conv_cuda("muffin_conv3d_forward");
}

int muffin_conv3d_backward_data(const void* d_dz, const float* d_w, const void* d_mask, void* d_da, int nz, int ny,
                                int nx, void* d_scratch, size_t scratch_bytes, cudaStream_t stream) {
  int r = layer_args(d_dz, d_da, nz, ny, nx, d_scratch, scratch_bytes);
  if (r != MUFFIN_OK) return r;
  if (!d_w) return conv_fail(MUFFIN_ERR_ARG, "NULL weights");
  if (d_mask && !aligned16(d_mask)) return conv_fail(MUFFIN_ERR_ARG, "mask must be 16-byte aligned");
  const Dims d = make_dims(nz, ny, nx);
  bf16* wk = (bf16*)d_scratch;
  k_pack_layer<<<(WMID + 255) / 256, 256, 0, stream>>>(d_w, wk, 1);
  launch_conv(EPI_MASK, (const bf16*)d_dz, wk, nullptr, (const bf16*)d_mask, (bf16*)d_da, d, sm_count(), stream);
  return conv_cuda("muffin_conv3d_backward_data");
}

int muffin_conv3d_backward_weights(const void* d_a, const void* d_dz, float* d_dw, float* d_db, int nz, int ny,
                                   int nx, void* d_scratch, size_t scratch_bytes, cudaStream_t stream) {
  int r = layer_args(d_a, d_dz, nz, ny, nx, d_scratch, scratch_bytes);
  if (r != MUFFIN_OK) return r;
  if (!d_dw) return conv_fail(MUFFIN_ERR_ARG, "NULL weight gradient");
  const Dims d = make_dims(nz, ny, nx);
  char* base = (char*)d_scratch + align256(WMID * 2);
  const int P = part_slots(d);
  float* part = (float*)base;
  float* bpart = (float*)(base + align256((size_t)P * WMID * 4));
  launch_wgrad_mid((const bf16*)d_a, (const bf16*)d_dz, part, bpart, d_dw, d_db, d, sm_count(), stream);
  return conv_cuda("muffin_conv3d_backward_weights");
}

const char* muffin_conv3d_last_error(void) { return g_conv_err.c_str(); }

}  // extern "C"
