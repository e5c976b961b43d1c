// The special-function unit's instructions in the forms that flush subnormal numbers to zero (PTX rsqrt, ex2 and
// rcp .approx.ftz.f32), for the ion-ion pass (no pair within reach has a subnormal distance, and a factor below
// 2^-126 is nothing) and the network's forward pass.  About eleven instructions per pair less than with the handling of subnormals.  Each is within
// 2^-22 of its result; e^x = 2^(x log2 e) adds the roundings of log2 e and of the product, 2^-24 of the exponent each,
// so |x| 2^-23 of the result.
#pragma once

namespace srbe {

__device__ __forceinline__ float rsqrt_n(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float exp_n(float x) {
  constexpr float kLog2E = (float)1.44269504088896340736;
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x * kLog2E));
  return r;
}
__device__ __forceinline__ float rcp_n(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// a / d from r, the reciprocal of d within 2^-22: the quotient's residual a - q d is exact in one FMA and corrects
// q (Newton's step for the quotient; Markstein, IBM J. Res. Dev. 34, 1990), so that only its own rounding is left,
// 2^-24.  For d and 1 / d normal, a finite and no underflow.
__device__ __forceinline__ float quotient(float a, float d, float r) {
  const float q = a * r;
  return fmaf(fmaf(-q, d, a), r, q);
}

}  // namespace srbe
