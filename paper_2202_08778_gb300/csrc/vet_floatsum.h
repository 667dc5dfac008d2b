// vet_floatsum.h -- sums of FP32 values to FP64's precision in FP32 arithmetic.
//
// GB300 executes two FP64 operations per clock per SM: an FP64 addition and the
// conversion before it hold the pipe for 32 clocks per warp, where the 13 FP32
// additions here take four.
#pragma once

#include <cuda_runtime.h>

namespace vet {

// s += x, returns the rounding of it, exactly (TwoSum, Knuth).  Explicitly rounded
// additions: an operand that is itself a product must not be contracted into them.
__device__ __forceinline__ float two_sum(float &s, float x) {
  const float r = __fadd_rn(s, x), t = __fsub_rn(r, s);
  const float e = __fadd_rn(__fsub_rn(s, __fsub_rn(r, t)), __fsub_rn(x, t));
  s = r;
  return e;
}

// A sum as three floats: two exact sums carry their roundings on, the third
// collects what is below 2^-48 of the total, so the result is within an FP64
// rounding of the exact sum (not finite where a value or the sum is not).
struct FloatSum {
  float a = 0.f, b = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float x) { c = __fadd_rn(c, two_sum(b, two_sum(a, x))); }
  // x + y, |y| below 2^-23 |x|
  __device__ __forceinline__ void add(float x, float y) {
    const float e = two_sum(b, two_sum(a, x));
    c = __fadd_rn(c, __fadd_rn(e, two_sum(b, y)));
  }
  __device__ __forceinline__ double value() const { return (double)a + ((double)b + (double)c); }
};

}  // namespace vet
