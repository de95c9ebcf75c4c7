// Compensated sums shared by the kernels.
#pragma once
#include <cuda_runtime.h>

namespace lpa {

// Error-free sum of two floats (Knuth's two-sum) and product (FMA residual).
__device__ __forceinline__ void comp_add(float &hi, float &lo, float a, float b) {
  float p = __fmul_rn(a, b);
  float pe = __fmaf_rn(a, b, -p);
  float s = __fadd_rn(hi, p);
  float bb = __fsub_rn(s, hi);
  float e = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bb)), __fsub_rn(p, bb));
  hi = s;
  lo = __fadd_rn(lo, __fadd_rn(e, pe));
}

// comp_add on two sums at once: hi + lo += a b in each half, every operation rounded as there
// (differences as products with -1; `na` is -a, so that the residual needs no negation).
__device__ __forceinline__ void comp_add2(float2 &hi, float2 &lo, float2 a, float2 na, float2 b) {
  const float2 M = make_float2(-1.f, -1.f);
  const float2 p = __fmul2_rn(a, b);
  const float2 npe = __ffma2_rn(na, b, p);  // -(a b - p)
  const float2 s = __fadd2_rn(hi, p);
  const float2 bb = __ffma2_rn(hi, M, s);
  const float2 e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, M, s), M, hi), __ffma2_rn(bb, M, p));
  hi = s;
  lo = __fadd2_rn(lo, __ffma2_rn(npe, M, e));
}

// The same for hi + lo += a: the product with 1 leaves nothing out.
__device__ __forceinline__ void comp_sum2(float2 &hi, float2 &lo, float2 a) {
  const float2 M = make_float2(-1.f, -1.f);
  const float2 s = __fadd2_rn(hi, a);
  const float2 bb = __ffma2_rn(hi, M, s);
  const float2 e = __fadd2_rn(__ffma2_rn(__ffma2_rn(bb, M, s), M, hi), __ffma2_rn(bb, M, a));
  hi = s;
  lo = __fadd2_rn(lo, e);
}

}  // namespace lpa
