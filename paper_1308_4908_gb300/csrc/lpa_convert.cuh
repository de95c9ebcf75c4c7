// Conversion of raw samples, shared by the reconstruction kernels and the conversion pass.
#pragma once
#include <stdint.h>

#include "lpa_launch.h"

// sensor-space positions are clamped to +-LPA_FAR px (far outside any sensor) before integer conversion
#define LPA_FAR 1.0e7
#define LPA_FAR_F 1.0e7f

namespace lpa {

// Staged sample layout: (f, 1/s2) (1/s for the printed weight); 1/s2 = 0 excludes the sample.
__device__ __forceinline__ float2 stage_pair(float f, float iv) { return make_float2(f, iv); }
__device__ __forceinline__ bool sample_ok(float2 fv) { return fv.y > 0.f; }
// The staged value of raw sample y at sensor pixel (X, Y), inside the frame: Eq. 18 and the inverse
// of Eq. 20 (its square root for the printed weight K / s); (0, 0) when saturated. `scalar`: the
// sensor has no per-pixel calibration frames.
template <bool LIT>
__device__ __forceinline__ float2 convert_sample(const LpaSensorK &Sk, bool scalar, int X, int Y, float y) {
  float f = 0.f, iv = 0.f;
  if (scalar) {
    if (y < Sk.sat) {
      const float e0 = y - Sk.black;
      f = e0 * Sk.inv_gtn;
      iv = __fdividef(Sk.gtn2, fmaf(Sk.gain, fmaxf(e0, 0.f), Sk.read_var));
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
      f = __fdividef(e0 * Sk.inv_gtn, a);
      iv = __fdividef(Sk.gtn2 * a * a, fmaf(Sk.gain, fmaxf(e0, 0.f), rv));
      if (LIT) iv = sqrtf(iv);
    }
  }
  return stage_pair(f, iv);
}

}  // namespace lpa
