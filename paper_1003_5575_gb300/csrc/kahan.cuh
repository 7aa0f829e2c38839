// Compensated (Kahan) FP32 summation, shared by the prediction and the adjoint.
#pragma once
#include "common.cuh"

namespace rts {

// compensated summation step: the running total is sum - comp
__device__ inline void kahan_add(float& sum, float& comp, float x) {
  const float y = x - comp;
  const float t = sum + y;
  comp = (t - sum) - y;
  sum = t;
}

// x into sum (two of them, packed); x is left with what the sum's rounding dropped, and
// the next x is added up on top of it
__device__ __forceinline__ void kahan_carry2(float2& sum, float2& x) {
  const float2 neg = make_float2(-1.f, -1.f), t = fadd2(sum, x);
  x = ffma2(neg, ffma2(neg, sum, t), x);
  sum = t;
}

// An unevaluated sum hi + lo of two floats.  Adding two of them costs 8 FP32
// instructions and keeps about 47 bits; an FP64 addition occupies a
// sub-partition's FP64 pipe for 64 cycles a warp.
struct FF { float hi, lo; };
__device__ __forceinline__ FF ff_two_sum(float a, float b) {
  FF r;
  r.hi = __fadd_rn(a, b);
  const float bb = __fsub_rn(r.hi, a);
  r.lo = __fadd_rn(__fsub_rn(a, __fsub_rn(r.hi, bb)), __fsub_rn(b, bb));
  return r;
}
__device__ __forceinline__ FF ff_add(FF a, FF b) {
  FF r = ff_two_sum(a.hi, b.hi);
  r.lo = __fadd_rn(r.lo, __fadd_rn(a.lo, b.lo));
  return r;
}
// s + a b, the product exact
__device__ __forceinline__ FF ff_fma(float a, float b, FF s) {
  const float p = __fmul_rn(a, b), e = fmaf(a, b, -p);
  FF r = ff_two_sum(s.hi, p);
  r.lo = __fadd_rn(r.lo, __fadd_rn(s.lo, e));
  return r;
}

}  // namespace rts
