// Conversion of raw samples, shared by the reconstruction kernels and the conversion pass.
#pragma once
#include <stdint.h>

#include "lpa_launch.h"
#include "lpa_ptx.cuh"

// sensor-space positions are clamped to +-LPA_FAR px (far outside any sensor) before integer conversion
#define LPA_FAR 1.0e7
#define LPA_FAR_F 1.0e7f

namespace lpa {

// Staged sample layout: (f, 1/s2) (1/s for the printed weight); 1/s2 = 0 excludes the sample.
__device__ __forceinline__ float2 stage_pair(float f, float iv) { return make_float2(f, iv); }
__device__ __forceinline__ bool sample_ok(float2 fv) { return fv.y > 0.f; }
// The staged value of raw sample y at sensor pixel (X, Y), inside the frame: Eq. 18 and the inverse
// of Eq. 20 (its square root for the printed weight K / s). An excluded sample is (0, 0), so that a window value of
// any size times it adds nothing: a saturated one, and one whose weight is 0 or whose value, weight or
// product FP32 cannot hold (a sensitivity or read variance decades beyond any sensor's, a bias that is
// no number). Sensors marked plain (`plain` = LpaSensorK::plain) have no such samples besides the saturated ones.
template <bool LIT>
__device__ __forceinline__ float2 convert_sample(const LpaSensorK &Sk, bool plain, int X, int Y, float y) {
  float f = 0.f, iv = 0.f;
  if (plain) {
    if (y < Sk.sat) {
      const float e0 = y - Sk.black;
      f = e0 * Sk.inv_gtn;
      iv = div_approx(Sk.gtn2, fmaf(Sk.gain, fmaxf(e0, 0.f), Sk.read_var));
      if (LIT) iv = sqrtf(iv);
    }
  } else {
    const long px = (long)Y * Sk.width + X;
    const float b = Sk.bias ? Sk.bias[px] : Sk.black;
    const float rv = Sk.rvar ? Sk.rvar[px] : Sk.read_var;
    const float sat = Sk.satf ? (float)Sk.satf[px] : Sk.sat;
    if (y < sat) {
      const float a = Sk.prnu ? Sk.prnu[px] : 1.f;
      const float e0 = y - b;
      f = __fdividef(e0 * Sk.inv_gtn, a);  // (denormal divisors too, unlike div_approx)
      iv = __fdividef(Sk.gtn2 * a * a, fmaf(Sk.gain, fmaxf(e0, 0.f), rv));
      if (LIT) iv = sqrtf(iv);
      if (!(iv > 0.f && fabsf(iv * f) <= 3.402823466e38f)) f = iv = 0.f;
    }
  }
  return stage_pair(f, iv);
}

// convert_sample<false> of two samples of a plain sensor, in paired arithmetic with
// its roundings: f and 1 / s2, which is 0 (f is not, unlike there) where ok is false or the sample is
// saturated.
__device__ __forceinline__ void convert_two(const LpaSensorK &S, float y0, float y1, bool ok0, bool ok1, float2 &f, float2 &iv) {
  const float2 e = __fadd2_rn(make_float2(y0, y1), make_float2(-S.black, -S.black));
  f = __fmul2_rn(e, make_float2(S.inv_gtn, S.inv_gtn));
  const float2 d = __ffma2_rn(make_float2(S.gain, S.gain), make_float2(fmaxf(e.x, 0.f), fmaxf(e.y, 0.f)),
                              make_float2(S.read_var, S.read_var));
  iv = make_float2(div_approx(S.gtn2, d.x), div_approx(S.gtn2, d.y));
  iv.x = y0 < S.sat && ok0 ? iv.x : 0.f;
  iv.y = y1 < S.sat && ok1 ? iv.y : 0.f;
}

}  // namespace lpa
