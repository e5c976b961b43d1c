// Small-angle part of the FP64 sine and cosine in integer arithmetic.
//
// GB300 issues 1.7 FP64 operations per clock and SM against 64 integer ones, so the reduced angle's
// cos x - 1 and sin x (|x| <= pi / 1024, the remainder of a 64-bit phase after its 10 table bits) are
// evaluated with 11 32 x 32 -> 64-bit multiplications and assembled into doubles by integer
// instructions; the FP64 pipe is left with the four multiply-adds of the angle addition.
#pragma once
#include <stdint.h>

#include "pairfix.cuh"

namespace srbe {

// hi 64 bits of a b (signed), without the product of the low halves' low part: within 3 units
__host__ __device__ __forceinline__ int64_t fix_mulhi(int64_t a, int64_t b) {
  const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32);
  const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);   // 31 bits
  return (int64_t)ah * bh + (((int64_t)ah * bl) >> 31) + (((int64_t)bh * al) >> 31);
}

// cos x - 1 and sin x for x = 2 pi rem / 2^64, |rem| <= 2^53.  With rho = rem / 2^53, q = rho^2 and
// delta = pi / 1024:
//   cos x - 1 = -q (delta^2 / 2) (1 - q delta^2 / 12)          (the next term is 1.2e-18)
//   sin x     = rho delta (1 - q (delta^2 / 6 - q delta^4 / 120))
__host__ __device__ __forceinline__ void small_cos_sin(int64_t rem, double &cm1, double &sx) {
  constexpr double kDelta = 3.14159265358979323846 / 1024.0, kD2 = kDelta * kDelta;
  constexpr double kTwo80 = 1208925819614629174706176.0, kTwo71 = 2361183241434822606848.0;
  constexpr int64_t kC2 = (int64_t)(kD2 / 2 * kTwo80);                          // Q80
  constexpr int32_t kC4 = (int32_t)(kD2 * kD2 / 24 * kTwo80 / 4096.0 + 0.5);    // Q68
  // delta in Q71: the double nearest to pi / 1024 is 1.2e-16 / 1024 short, which shows at 2^-71
  constexpr int64_t kS1 = (int64_t)(kDelta * kTwo71) + (int64_t)(1.2246467991473532e-16 / 1024.0 * kTwo71 + 0.5);
  constexpr int32_t kS3 = (int32_t)(kD2 * kDelta / 6 * kTwo71 / 8192.0 + 0.5);  // Q58
  constexpr int32_t kS5 = (int32_t)(kD2 * kD2 * kDelta / 120 * kTwo71 / 8192.0 + 0.5);   // Q58
  const int64_t r = rem << 10;                                                  // rho in Q63
  const int32_t rh = (int32_t)(r >> 32), rl = (int32_t)((uint32_t)r >> 1);
  const int64_t q = (int64_t)rh * rh + (((int64_t)rh * rl) >> 30);              // rho^2 in Q62
  const int32_t qh = (int32_t)(q >> 32);                                        // Q30
  const int64_t k = kC2 - (((int64_t)qh * kC4) >> 18);                          // (delta^2 / 2)(1 - ...), Q80
  cm1 = -fix_to_double(fix_mulhi(q, k), -78);
  const int32_t f = kS3 - (int32_t)(((int64_t)qh * kS5) >> 30);
  const int64_t b = kS1 - (((int64_t)qh * f) >> 17);                            // delta (1 - ...), Q71
  sx = fix_to_double(fix_mulhi(r, b), -70);
}

}  // namespace srbe
