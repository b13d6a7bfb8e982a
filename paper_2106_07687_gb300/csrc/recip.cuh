// Reciprocals from the hardware's approximation by Newton's iteration, in place
// of the compiled divisions, which branch (FP32) and take a dozen FP64
// instructions (each 64 cycles of a warp's scheduler on this GPU).  The last step
// from an approximation good to half of the bits and more rounds like a division
// (P. Markstein, "Computation of elementary functions on the IBM RISC System/6000
// processor", 1990); tests/test_gpu_recip.py compares both with division.
#pragma once
#include <cuda_runtime.h>

namespace dnnmg {

// 1 / x for x >= 1: 1.0f / x for every float in [1, 2^125); above, where x may be
// infinite, the approximation itself, below 2^-124.
__device__ __forceinline__ float recip_ge1(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  const float r = __fmaf_rn(y, __fmaf_rn(-x, y, 1.0f), y);
  return x < 0x1p125f ? r : y;
}

// 1 / d to within one unit in the last place of the rounded quotient, for normal d
// with a normal reciprocal (two steps from about 20 bits: the error before the last
// rounding is 2^-80 of the value); NaN for d infinite, zero or subnormal.
__device__ __forceinline__ double recip64(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
#pragma unroll
  for (int k = 0; k < 2; ++k) y = fma(y, fma(-d, y, 1.0), y);
  return y;
}

// The same, and by the approximation 0 for d infinite or above 2^1022 and infinity
// for d zero or subnormal.
__device__ __forceinline__ double recip64_any(double d) {
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(d));
  const unsigned e = (unsigned)__double2hiint(y) & 0x7FF00000u;
  const double r = recip64(d);
  return e - 1u < 0x7FEFFFFFu ? r : y;  // e is neither 0 nor 0x7FF00000
}

}  // namespace dnnmg
