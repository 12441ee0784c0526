// Reciprocals and inverse square roots without the IEEE division's and square root's
// instruction sequences.  On GB300 an FP64 instruction occupies its pipe for 16 cycles a
// warp, so the FP64 kernels, bound by that pipe, take the hardware's approximation and
// two or three fused multiply-adds.  Third-order iterations of Householder (The Numerical
// Treatment of a Single Nonlinear Equation, 1970) on 1 / y - x and 1 / y^2 - x: with the
// remainder e = 1 - x r or 1 - x y^2 the next value is r (1 + e + e^2) or
// y (1 + e / 2 + 3 e^2 / 8), off by the order of e^3.  The approximations' e is below 2^-19,
// so what is left is the rounding of the last steps.  tests/test_reciprocal.py compares
// them with CUDA's 1 / x and 1 / sqrt(x) over the exponents.
#pragma once
#include <cuda_runtime.h>

namespace lbmk {

// 1 / x for x and 1 / x in the normal range, within one unit in the last place (FP32: one
// Newton step).
__device__ __forceinline__ float recip(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return fmaf(r, fmaf(-x, r, 1.0f), r);
}
__device__ __forceinline__ double recip(double x) {
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(x));
  const double e = fma(-x, r, 1.0);
  return fma(r, fma(e, e, e), r);
}

// 1 / x where the approximation as it is (within two units in the last place) is enough in
// FP32; FP64 as above.
__device__ __forceinline__ float rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ double rcp(double x) { return recip(x); }

// 1 / |g| for g2 = |g|^2 > 0, else 0; within two units in the last place.
__device__ __forceinline__ float inv_norm(float g2) { return g2 != 0.0f ? rsqrtf(g2) : 0.0f; }
__device__ __forceinline__ double inv_norm(double g2) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(g2));
  const double e = fma(-g2 * y, y, 1.0);
  y = fma(y * e, fma(e, 0.375, 0.5), y);
  return g2 > 1e-300 ? y : 0.0;  // a smaller |g|^2 has left the normal range
}

}  // namespace lbmk
