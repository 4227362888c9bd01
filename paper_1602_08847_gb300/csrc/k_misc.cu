// Small kernels: deterministic FP64 reductions, the power-method helpers,
// a counter-based start vector, and the plane permutation between the natural
// and the class-permuted layouts of U.
#include "device.cuh"
#include "exact_sum.cuh"
#include "internal.h"

namespace muffin {

// One block sums (op 0) or maxes (op 1) n partials in a fixed order.
__global__ void __launch_bounds__(1024) k_reduce_partials(const double* __restrict__ p, int n, double* out, int op) {
  __shared__ double red[32];
  double acc = 0.0;
  for (int i = threadIdx.x; i < n; i += blockDim.x) acc = op == 0 ? acc + p[i] : fmax(acc, p[i]);
  if (op == 0) {
    acc = block_sum(acc, red);
  } else {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc = fmax(acc, __shfl_down_sync(0xffffffffu, acc, o));
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
    __syncthreads();
    if (threadIdx.x < 32) {
      acc = threadIdx.x < (blockDim.x + 31) / 32 ? red[threadIdx.x] : 0.0;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc = fmax(acc, __shfl_down_sync(0xffffffffu, acc, o));
    }
  }
  if (threadIdx.x == 0) *out = acc;
}

// FP64 runs at 1/64 of the FP32 rate here: the conversions and the double
// multiply-add of every value, and a square root and division in every thread
// of the scaling, bound these two kernels of the power method at 404 and 406 us
// for 67 M values; 95 and 90 us so.  Products are split exactly into two floats
// and summed in three (Sum3) over 16 values, then added to the double: three
// roundings to double where every value had one (float pairs, 60 us, lost the
// bits past 48).  A group with a product outside the range in which that is
// exact is summed in double.
__global__ void __launch_bounds__(256) k_dot(const float* __restrict__ a, const float* __restrict__ b, size_t n,
                                            double* partials) {
  __shared__ double red[32];
  double acc = 0.0;
  const size_t n4 = (((uintptr_t)a | (uintptr_t)b) & 15) == 0 ? n / 4 : 0, step = (size_t)gridDim.x * blockDim.x;
  const size_t first = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  for (size_t i = first; i < n4; i += 4 * step) {
    float x[16], y[16];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const size_t j = i + e * step;
      float4 u = make_float4(0.f, 0.f, 0.f, 0.f), v = u;
      if (j < n4) {
        u = __ldg(reinterpret_cast<const float4*>(a) + j);
        v = __ldg(reinterpret_cast<const float4*>(b) + j);
      }
      x[4 * e] = u.x; x[4 * e + 1] = u.y; x[4 * e + 2] = u.z; x[4 * e + 3] = u.w;
      y[4 * e] = v.x; y[4 * e + 1] = v.y; y[4 * e + 2] = v.z; y[4 * e + 3] = v.w;
    }
    Sum3 s;
    bool exact = true;
#pragma unroll
    for (int e = 0; e < 16; ++e) {
      const float m = fabsf(__fmul_rn(x[e], y[e]));
      exact = exact && ((m >= 1e-28f && m <= 1e30f) || x[e] == 0.f || y[e] == 0.f);
      s.add_product(x[e], y[e]);
    }
    if (exact) {
      s.into(acc);
    } else {
#pragma unroll 1
      for (int e = 0; e < 4; ++e) {
        const size_t j = i + e * step;
        if (j >= n4) break;
        for (int q = 0; q < 4; ++q) acc += (double)a[4 * j + q] * (double)b[4 * j + q];
      }
    }
  }
  for (size_t i = 4 * n4 + first; i < n; i += step) acc += (double)a[i] * (double)b[i];
  acc = block_sum(acc, red);
  if (threadIdx.x == 0) partials[blockIdx.x] = acc;
}

__device__ __noinline__ float4 scale4_double(float4 v, double f) {   // a call: seldom taken
  return make_float4((float)(v.x * f), (float)(v.y * f), (float)(v.z * f), (float)(v.w * f));
}

// x <- (float)(x * num / sqrt(den))   (num == nullptr: factor 1); the factor is
// formed once a block, and where it is two floats the values are rounded through
// them (scale_float), the few it cannot tell in double.  67 M values: 90 us
__global__ void k_scale(float* x, size_t n, const double* num, const double* den) {
  __shared__ double s_f;
  __shared__ float s_hi, s_lo;
  if (threadIdx.x == 0) {
    s_f = (num ? *num : 1.0) / sqrt(*den);
    s_hi = (float)s_f;
    s_lo = (float)(s_f - (double)s_hi);
  }
  __syncthreads();
  const size_t step = (size_t)gridDim.x * blockDim.x, first = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  const float hi = s_hi, lo = s_lo;
  if (hi >= 1e-30f && hi <= 1e30f) {
    const size_t n4 = ((uintptr_t)x & 15) == 0 ? n / 4 : 0;
    float4* x4 = reinterpret_cast<float4*>(x);
#pragma unroll 2
    for (size_t i = first; i < n4; i += step) {
      const float4 v = x4[i];
      float4 r;
      const bool a = scale_float(v.x, hi, lo, &r.x), b = scale_float(v.y, hi, lo, &r.y);
      const bool c = scale_float(v.z, hi, lo, &r.z), d = scale_float(v.w, hi, lo, &r.w);
      if (!(a && b && c && d)) r = scale4_double(v, s_f);
      x4[i] = r;
    }
    for (size_t i = 4 * n4 + first; i < n; i += step) x[i] = (float)(x[i] * s_f);
  } else {
    for (size_t i = first; i < n; i += step) x[i] = (float)(x[i] * s_f);
  }
}

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014) of (seed + index): uniform in [-1, 1).
__device__ __forceinline__ uint64_t splitmix64(uint64_t z) {
  z += 0x9e3779b97f4a7c15ull;
  z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
  z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
  return z ^ (z >> 31);
}

__global__ void k_fill_random(float* x, size_t n, uint64_t seed) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const uint64_t r = splitmix64(seed * 0x100000001b3ull + i);
    x[i] = (float)((double)(r >> 11) * (2.0 / 9007199254740992.0) - 1.0);
  }
}

// Planes j >= j1 of U between natural (to_class = 0) and class-permuted layout.
__global__ void k_permute(const float* __restrict__ src, float* __restrict__ dst, int n, int L, int J, int j1,
                          int to_class) {
  const size_t P = (size_t)n * n;
  const size_t total = (size_t)L * (J + 1) * P;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    const size_t plane = i / P;
    const int j = (int)(plane % (J + 1));
    const int p = (int)(i % P);
    const int lgs = j >= j1 ? j1 : 0;
    const int ci = class_index(p / n, p % n, n, lgs);
    if (to_class) dst[plane * P + ci] = src[i];
    else dst[i] = src[plane * P + ci];
  }
}

__global__ void k_nonfinite(const float* __restrict__ x, size_t n, int* count) {
  int c = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    c += isfinite(x[i]) ? 0 : 1;
  c = warp_sum(c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(count, c);
}

static int grid_for(size_t n, int block, int cap) {
  size_t g = (n + block - 1) / block;
  if (g > (size_t)cap) g = cap;
  return g < 1 ? 1 : (int)g;
}

cudaError_t launch_sum_partials(const double* partials, int n, double* out, cudaStream_t s) {
  k_reduce_partials<<<1, 1024, 0, s>>>(partials, n, out, 0);
  return cudaGetLastError();
}

cudaError_t launch_max_partials(const double* partials, int n, double* out, cudaStream_t s) {
  k_reduce_partials<<<1, 1024, 0, s>>>(partials, n, out, 1);
  return cudaGetLastError();
}

cudaError_t launch_dot(const float* a, const float* b, size_t n, double* partials, int* nparts, cudaStream_t s) {
  const int g = grid_for(n / 16 + 1, 256, 1024);
  *nparts = g;
  k_dot<<<g, 256, 0, s>>>(a, b, n, partials);
  return cudaGetLastError();
}

cudaError_t launch_scale(float* x, size_t n, const double* num, const double* den, cudaStream_t s) {
  k_scale<<<grid_for(n / 4 + 1, 256, 2048), 256, 0, s>>>(x, n, num, den);
  return cudaGetLastError();
}

cudaError_t launch_fill_random(float* x, size_t n, uint64_t seed, cudaStream_t s) {
  k_fill_random<<<grid_for(n, 256, 4096), 256, 0, s>>>(x, n, seed);
  return cudaGetLastError();
}

cudaError_t launch_permute_planes(const float* src, float* dst, int n, int L, int J, int j1, int to_class,
                                  cudaStream_t s) {
  const size_t total = (size_t)L * (J + 1) * n * n;
  k_permute<<<grid_for(total, 256, 8192), 256, 0, s>>>(src, dst, n, L, J, j1, to_class);
  return cudaGetLastError();
}

cudaError_t launch_nonfinite_count(const float* x, size_t n, int* count, cudaStream_t s) {
  k_nonfinite<<<grid_for(n, 256, 4096), 256, 0, s>>>(x, n, count);
  return cudaGetLastError();
}

}  // namespace muffin
