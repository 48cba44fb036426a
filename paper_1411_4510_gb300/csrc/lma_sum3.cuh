// Sums with FP64's accuracy in FP32 instructions.
//
// An FP64 instruction occupies a scheduler for 64 clocks (and so does the conversion of an FP32 operand), an FP32 one
// for one.  A running sum in three floats takes a product in 22 of them.  After n products the middle part is at most
// (n + 1) 2^-24 of the terms' magnitudes, the last one 2 n (n + 1) 2^-48 and its rounding errors 4 n^2 (n + 1) 2^-72,
// less than FP64's n 2^-53 up to kSum3Terms = 256, wherever no part leaves a float's range.  The callers check that on
// the result and add in FP64 otherwise, so that infinities, NaN and tiny values come out as FP64 has them.
#pragma once
#include <cuda_runtime.h>

namespace lma {

constexpr int kSum3Terms = 256;  // a lane's

// a + b = s + e exactly (Knuth's TwoSum); s replaces a, e is returned.
__device__ __forceinline__ float two_sum_in(float& a, float b) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  const float e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  a = s;
  return e;
}

struct Sum3 {
  float h = 0.f, m = 0.f, l = 0.f;
  __device__ __forceinline__ void add(float x) {
    const float e = two_sum_in(h, x);
    l = __fadd_rn(l, two_sum_in(m, e));
  }
  __device__ __forceinline__ void add_product(float a, float b) {
    const float p = __fmul_rn(a, b);
    add(p);
    l = __fadd_rn(l, two_sum_in(m, __fmaf_rn(a, b, -p)));
  }
  // a (b.x + b.y + b.z), b a double in three floats (k_split_beta); the errors are 15 n^3 2^-72: half as many terms
  __device__ __forceinline__ void add_product(float a, float4 b) {
    add_product(a, b.x);
    const float p = __fmul_rn(a, b.y);
    l = __fadd_rn(l, two_sum_in(m, p));
    l = __fadd_rn(l, __fmaf_rn(a, b.z, __fmaf_rn(a, b.y, -p)));
  }
  __device__ __forceinline__ double value() const { return (double)h + ((double)m + (double)l); }
};

// Whether a sum of products held in Sum3 stands: finite (an infinity or an overflow turns the parts into NaN), and so far
// above what underflow can have cost (2^-150 a term, 2^32 terms at most) that this is less than an FP64 rounding.
__device__ __forceinline__ bool sum3_stands(double v) { return fabs(v) >= 0x1p-64; }

// The sum of a few terms, rounded once; false if the value is too close to a tie to tell or not finite: the caller then
// adds in FP64.
__device__ __forceinline__ bool sum3_round(const Sum3& s, float& out) {
  float h = s.h, m = s.m, l = s.l;
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    l = two_sum_in(m, l);
    m = two_sum_in(h, m);
  }
  // h + m is rounded to h; l is less than half of m's last place (at most that, with m a tie, where l is not zero)
  out = h;
  return l == 0.f || __fmaf_rn(m, 1.0001f, h) == h;
}

// The warp's sum of v, in every lane.
__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

}  // namespace lma
