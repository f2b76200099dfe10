// Wave speeds in FP32 that decide for which points the FP64 stages evaluate
// the FP64 speed: only those whose FP32 one comes within 2^-9 of the tile's
// largest. So that none of them can hide the maximum, every value here is
// within 2^-11 (relative) of the speed from both sides, or NaN: where FP32
// cannot tell, the FP64 speed is evaluated.
#pragma once

#include "hweno.h"
#include "weno_df.cuh"

namespace hweno {

// Euler: sound speed from rho, its reciprocal, E and the kinetic energy.
// NaN for p below 2^-8 E, where the subtraction costs too many bits, and for
// rho, E outside 2^-50 .. 2^50 (or a sound speed beyond 2^50), where a product
// could leave the normal range; for gamma - 1 below 2^-10, which FP32 rounds.
__device__ __forceinline__ float rough_sound(float r, float ir, float E, float kin, float gam) {
  const float e = E - kin, c2 = gam * (gam - 1.f) * e * ir;
  const bool ok = e >= 0.00390625f * E && E >= 0x1p-50f && E <= 0x1p50f && r >= 0x1p-50f &&
                  r <= 0x1p50f && c2 <= 0x1p100f && gam >= 1.f + 0x1p-10f;
  return ok ? sqrtf(c2) : __int_as_float(0x7fc00000);
}

template <int EQ>
__device__ __forceinline__ float rough_speed(const double* u, float gam) {
  if constexpr (EQ == HWENO_BURGERS) {
    return fabsf(to_float(u[0]));
  } else if constexpr (EQ == HWENO_BUCKLEY) {
    // (1 - u before the conversion: next to u = 1 its bits are u's last)
    const float x = to_float(u[0]), y = to_float(sub(1.0, u[0])), D = 4.f * x * x + y * y;
    return fabsf(x) <= 0x1p15f ? fabsf(8.f * x * y) / (D * D) : __int_as_float(0x7fc00000);
  } else {
    const float r = to_float(u[0]), m = to_float(u[1]), ir = 1.f / r, vel = m * ir;
    return fabsf(vel) + rough_sound(r, ir, to_float(u[2]), 0.5f * m * vel, gam);
  }
}

// The same of both directions of a 2D state. Velocities before the kinetic
// energy: squares of small momenta would fall under the FP32 range.
template <int EQ>
__device__ __forceinline__ void rough_speeds2(const double* u, float gam, float& sx, float& sy) {
  if constexpr (EQ == HWENO_BURGERS) {
    sx = sy = fabsf(to_float(u[0]));
  } else {
    const float r = to_float(u[0]), m = to_float(u[1]), n = to_float(u[2]), ir = 1.f / r;
    const float vx = m * ir, vy = n * ir;
    const float c = rough_sound(r, ir, to_float(u[3]), 0.5f * (m * vx + n * vy), gam);
    sx = fabsf(vx) + c;
    sy = fabsf(vy) + c;
  }
}

}  // namespace hweno
