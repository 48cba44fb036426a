// Arithmetic on pairs of floats.
//
// Numbers held as the sum of two floats (48 bits): an FP64 instruction occupies a
// scheduler for 64 clocks, a float one for one, so where FP64 is more than the result
// needs but a float is less, sums and products of pairs are 5 to 10 times cheaper.
#pragma once
#include <cuda_runtime.h>

namespace lma {

struct Pair2 {
  float h, l;
};
__device__ __forceinline__ Pair2 quick2(float a, float b) {  // |a| >= |b|
  const float s = __fadd_rn(a, b);
  return {s, __fsub_rn(b, __fsub_rn(s, a))};
}
__device__ __forceinline__ Pair2 sum2(float a, float b) {  // exact
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t))};
}
__device__ __forceinline__ Pair2 add2(Pair2 a, Pair2 b) {
  const Pair2 s = sum2(a.h, b.h);
  return quick2(s.h, __fadd_rn(s.l, __fadd_rn(a.l, b.l)));
}
__device__ __forceinline__ Pair2 mul2(Pair2 a, Pair2 b) {
  const float p = __fmul_rn(a.h, b.h);
  float e = __fmaf_rn(a.h, b.h, -p);
  e = __fmaf_rn(a.h, b.l, e);
  e = __fmaf_rn(a.l, b.h, e);
  return quick2(p, e);
}
__device__ __forceinline__ Pair2 scale2(Pair2 a, float b) {
  const float p = __fmul_rn(a.h, b);
  return quick2(p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p)));
}
__device__ __forceinline__ Pair2 split2(double x) {
  const float h = (float)x;
  return {h, (float)(x - (double)h)};
}
// acc += a b, the product and the sum exact but for the pair's last bits
__device__ __forceinline__ void fma2(Pair2& acc, float a, float b) {
  const float p = __fmul_rn(a, b);
  const Pair2 s = sum2(acc.h, p);
  acc = {s.h, __fadd_rn(acc.l, __fadd_rn(s.l, __fmaf_rn(a, b, -p)))};
}
// The warp's sum, in every lane.
__device__ __forceinline__ Pair2 warp_sum2(Pair2 v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    v = add2(v, Pair2{__shfl_xor_sync(0xffffffffu, v.h, o), __shfl_xor_sync(0xffffffffu, v.l, o)});
  return v;
}
__device__ __forceinline__ double to_double(Pair2 v) { return (double)v.h + (double)v.l; }

}  // namespace lma
