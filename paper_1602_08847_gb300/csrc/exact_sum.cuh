// Double results by float arithmetic.  Double arithmetic runs at 1/64 of the
// float rate here, so long sums add a few terms in floats between two additions
// to a double, by error-free steps, so that no bit is lost that a double would
// have held; and a product that is rounded to float in the end is formed in two.
#pragma once
#include <cuda_runtime.h>

namespace muffin {

// Three floats.  add() is Knuth's two-sum into hi, and of its rounding error
// into mid; what is left of that goes to lo in plain float32.  For the 32 terms
// or fewer that are added between two calls of into(), lo is below 2^-42 of the
// largest partial sum and its own rounding below 2^-61 of it, where a double
// rounds every addition to 2^-53.  The operations are the _rn intrinsics: the
// compiler may merge a plain * and + into one multiply-add, after which the
// "error" of a sum or of a product is another number.
// Needs |terms| and their sums within the range of floats, and terms of at least
// 2^-149 * 2^24 where their errors are to be exact: see the callers.
struct Sum3 {
  float hi = 0.f, mid = 0.f, lo = 0.f;

  // s <- s + x, the rounding error returned
  static __device__ __forceinline__ float two_sum(float& s, float x) {
    const float t = __fadd_rn(s, x), b = __fsub_rn(t, s);
    const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(t, b)), __fsub_rn(x, b));
    s = t;
    return e;
  }
  __device__ __forceinline__ void add(float x) { add_small(two_sum(hi, x)); }
  // a term of the size of hi's rounding errors
  __device__ __forceinline__ void add_small(float x) { lo = __fadd_rn(lo, two_sum(mid, x)); }
  // x * y, exactly
  __device__ __forceinline__ void add_product(float x, float y) {
    const float p = __fmul_rn(x, y);
    add(p);
    add_small(__fmaf_rn(x, y, -p));
  }
  __device__ __forceinline__ void into(double& acc) const {
    acc += (double)hi;
    acc += (double)mid;
    acc += (double)lo;
  }
};

// (float)((double)x * f) without double arithmetic, for f = hi + lo to 2^-48 of
// itself and 1e-30 <= hi <= 1e30: x f is formed in two floats, p + t, with an
// error below 2^-24 |t| + 2^-47 |p|; where p + (t - w) and p + (t + w) round to
// the same float for twice that as w, so does x f, and so does x f rounded to
// double first.  False where they differ (7 values in 10^7) or a term leaves the
// range of floats.
__device__ __forceinline__ bool scale_float(float x, float hi, float lo, float* out) {
  const float p = __fmul_rn(x, hi), m = fabsf(p);
  const float t = __fmaf_rn(x, lo, __fmaf_rn(x, hi, -p));
  const float w = __fmaf_rn(m, 0x1p-46f, fabsf(t) * 0x1p-22f);
  const float a = __fadd_rn(p, __fsub_rn(t, w)), b = __fadd_rn(p, __fadd_rn(t, w));
  *out = a;
  if (x == 0.f) *out = x;
  return x == 0.f || (a == b && m >= 0x1p-90f && m <= 0x1p120f);
}

}  // namespace muffin
