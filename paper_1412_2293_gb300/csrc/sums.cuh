// Sums of floats that carry more bits than FP64, on the FP32 pipe.
#pragma once

namespace qs {

// A running sum in three floats: each addition's rounding error, exactly
// (Knuth's two-sum), goes into the second float and that one's into the third,
// the cascaded summation of Ogita, Rump and Oishi (SIAM J. Sci. Comput. 26,
// 2005) with K = 3: as accurate as a sum in 72 bits, FP64's is one in 53.  A
// product enters as its rounded value and the exact remainder.  One is 22 FP32
// instructions; the FP64 multiply-add and its two conversions hold a
// scheduler's FP64 unit for about 64 cycles each on GB300.
// The exponents are FP32's: what overflows is infinite or NaN in value(), and a
// remainder below 2^-149 is lost.
struct Sum3 {
  float s = 0.f, c = 0.f, d = 0.f;
  static __device__ __forceinline__ float two_sum(float& a, float b) {
    const float t = __fadd_rn(a, b), z = __fadd_rn(t, -a);
    const float e = __fadd_rn(__fadd_rn(a, -__fadd_rn(t, -z)), __fadd_rn(b, -z));
    a = t;
    return e;
  }
  __device__ __forceinline__ void add(float v) { d = __fadd_rn(d, two_sum(c, two_sum(s, v))); }
  __device__ __forceinline__ void add(float a, float b) {
    const float p = __fmul_rn(a, b);
    add(p);
    d = __fadd_rn(d, two_sum(c, __fmaf_rn(a, b, -p)));
  }
  __device__ __forceinline__ double value() const { return (double)s + ((double)c + (double)d); }
};

}  // namespace qs
