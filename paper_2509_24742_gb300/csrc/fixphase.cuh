// The FP64 sine and cosine of a fixed-point phase in integer arithmetic.
//
// GB300 issues 1.7 FP64 operations per clock and SM against 64 integer ones, so the sine and cosine of a
// 64-bit phase are integer arithmetic to the end: the top 10 bits select a table angle (cos, sin in Q62),
// the remainder's cos x - 1 and sin x (|x| <= pi / 1024) take 11 32 x 32 -> 64-bit multiplications, the
// angle addition 12 more, and the two results are assembled into doubles by integer instructions.
#pragma once
#include <stdint.h>

#include "pairfix.cuh"

namespace srbe {

// 1 - cos x in Q78 and sin x in Q70 for x = 2 pi rem / 2^64, |rem| <= 2^53.  With rho = rem / 2^53, q = rho^2 and
// delta = pi / 1024:
//   cos x - 1 = -q (delta^2 / 2) (1 - q delta^2 / 12)          (the next term is 1.2e-18)
//   sin x     = rho delta (1 - q (delta^2 / 6 - q delta^4 / 120))
__host__ __device__ __forceinline__ void small_cos_sin(int64_t rem, int64_t &cm1, int64_t &sx) {
  constexpr double kDelta = 3.14159265358979323846 / 1024.0, kD2 = kDelta * kDelta;
  constexpr double kTwo80 = 1208925819614629174706176.0, kTwo71 = 2361183241434822606848.0;
  constexpr int64_t kC2 = (int64_t)(kD2 / 2 * kTwo80);                          // Q80
  constexpr int32_t kC4 = (int32_t)(kD2 * kD2 / 24 * kTwo80 / 4096.0 + 0.5);    // Q68
  // delta in Q71: the double nearest to pi / 1024 is 1.2e-16 / 1024 short, which shows at 2^-71
  constexpr int64_t kS1 = (int64_t)(kDelta * kTwo71) + (int64_t)(1.2246467991473532e-16 / 1024.0 * kTwo71 + 0.5);
  constexpr int32_t kS3 = (int32_t)(kD2 * kDelta / 6 * kTwo71 / 8192.0 + 0.5);  // Q58
  constexpr int32_t kS5 = (int32_t)(kD2 * kD2 * kDelta / 120 * kTwo71 / 8192.0 + 0.5);   // Q58
  const int64_t r = rem * 1024;                                                 // rho in Q63
  const int32_t rh = (int32_t)(r >> 32), rl = (int32_t)((uint32_t)r >> 1);
  const int64_t q = (int64_t)rh * rh + (((int64_t)rh * rl) >> 30);              // rho^2 in Q62
  const int32_t qh = (int32_t)(q >> 32);                                        // Q30
  const int64_t k = kC2 - (((int64_t)qh * kC4) >> 18);                          // (delta^2 / 2)(1 - ...), Q80
  cm1 = fix_mulhi(q, k);
  const int32_t f = kS3 - (int32_t)(((int64_t)qh * kS5) >> 30);
  const int64_t b = kS1 - (((int64_t)qh * f) >> 17);                            // delta (1 - ...), Q71
  sx = fix_mulhi(r, b);
}

// cos and sin of 2 pi th / 2^64; T: the table angle's (cos, sin) in Q62
__host__ __device__ __forceinline__ unsigned phase_index(uint64_t th) { return (unsigned)((th + (1ull << 53)) >> 54); }
__host__ __device__ __forceinline__ void phase_cos_sin(uint64_t th, longlong2 T, double &c, double &s) {
  // (th + 2^53) mod 2^54 - 2^53
  const int64_t rem = (int64_t)((th + (1ull << 53)) & ((1ull << 54) - 1)) - (1ll << 53);
  int64_t cm, sx;
  small_cos_sin(rem, cm, sx);
  // T (1 - cm) -+ T' sx: Q62 Q78 -> Q76, Q62 Q70 -> Q68
  c = fix_to_double(T.x - (fix_mulhi(T.x, cm) >> 14) - (fix_mulhi(T.y, sx) >> 6), -62);
  s = fix_to_double(T.y - (fix_mulhi(T.y, cm) >> 14) + (fix_mulhi(T.x, sx) >> 6), -62);
}

}  // namespace srbe
