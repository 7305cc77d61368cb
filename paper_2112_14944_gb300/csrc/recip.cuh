// Reciprocals and reciprocal square roots of the layout kernels: the
// special-function unit's estimate and correction steps from the residual.
// Where they are used they stand in a chain (the pivots) or on GB300's narrow
// FP64 pipe, and CUDA's functions take longer: k = 1,999, FP32 layout of 30
// updates, 1.45 ms with __frcp_rn, 1.41 so; k = 1,000 in FP64, 300 updates and
// the DPPR, 21.05 ms with __drcp_rn and rsqrt, 20.7 so.
#pragma once

#include <stdint.h>

namespace pprviz {

// 1 / a of a pivot in FP32: the estimate and one Newton step, for a and 1 / a
// normal. (The pivots of L^w + J / k: J / k has the eigenvalue 1, and an inverse
// in FP32 means something up to a condition of ~2^24, so they lie within
// 2^-24 .. 2^24.)
__device__ __forceinline__ float rcp_pos(float a) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return fmaf(fmaf(-a, r, 1.0f), r, r);
}

// The same in FP64: the estimate holds 20 bits or more, so two steps.
__device__ __forceinline__ double rcp_pos(double a) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(a));
  r = fma(fma(-a, r, 1.0), r, r);
  return fma(fma(-a, r, 1.0), r, r);
}

// 1 / sqrt(d2), 0 for d2 = 0: the estimate (20 bits or more) and one third-order
// step of the series of (1 - e)^-1/2, e = 1 - d2 y^2 (Halley's iteration): five
// FP64 operations, where a square root and a division take some tens. Values
// outside the normal range, infinities and NaN take the plain formula.
__device__ __forceinline__ double rsqrt_pos(double d2) {
  const uint32_t hi = (uint32_t)__double2hiint(d2);
  if (hi - 0x01000000u >= 0x7e000000u - 0x01000000u) return d2 > 0.0 ? 1.0 / sqrt(d2) : 0.0;
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d2));
  const double e = fma(-(d2 * y), y, 1.0);
  return fma(fma(e, 0.375, 0.5), e * y, y);
}

}  // namespace pprviz
