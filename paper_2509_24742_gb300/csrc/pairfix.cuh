// FP64 pair terms on few FP64 instructions (the FP64 form's real-space sums).
//
// GB300 issues 1.7 FP64 FMAs per clock and SM against 64 integer and 128 FP32 operations, so a pair
// written with sqrt, erfc, exp and divisions (about 150 FP64 instructions) costs 90 clocks of an SM.
// Here the geometry is integer arithmetic, the smooth factors are table polynomials in r^2, and 17
// FP64 FMAs are left:
//  * coordinates are 64-bit fixed-point fractions of a power-of-two period W >= 8 (rc + margin), so
//    differences (and image shifts) are exact modulo W and every pair within reach has |d| < W / 8 =: R1;
//  * S = r^2 in units of R1^2 2^-63 is formed from 31-bit limbs and rounded once;
//  * S is normalised: its exponent (12 octaves, r >= R1 / 64) and the next 7 bits select an interval, the
//    rest is t in [-1, 1); the radial factor is c0 + t (c1 + ... + t c7), c0..c3 in FP64, the tail in
//    FP32 (its terms are below 2^-30 of c0, so their FP32 rounding is below 2^-53);
//  * 1 / S comes from an FP32 reciprocal and one cubic Newton step (LJ powers);
//  * int64 -> double conversions are assembled with integer instructions.
// A pair closer than R1 / 64 leaves the table and takes the plain FP64 functions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace srbe {

constexpr int kPtOctaves = 12, kPtBits = 7;                // table intervals: 12 octaves of S, 128 each
constexpr int kPtSize = kPtOctaves << kPtBits;
constexpr uint64_t kPtMin = 1ull << (63 - kPtOctaves);     // smallest S of the table

struct __align__(16) PairCoef {                            // radial factor on one interval
  double c0, c1, c2, c3;
  float c4, c5, c6, c7;
};

// The Taylor expansion (in units of the half interval) of the radial factors around the centre of
// interval i: with s = r^2, f = erfc(a sqrt s) / sqrt s and E = exp(-a^2 s), df/ds = -g / 2 where
// g = (f + (2 a / sqrt pi) E) / s is the force factor -phi'(r) / r, so the Taylor coefficients of f and
// g follow from one another term by term:
//   f_{n+1} = -g_n / (2 (n + 1)),   g_n = (f_n + (2 a / sqrt pi) E_n - g_{n-1}) / s0.
// The interval is 2^-8 of its s on either side; the first term left out is below 1e-17 of c0.
struct RadialTaylor {
  double f[8], g[8];
};
__host__ __device__ inline void radial_taylor(double s0, double a, double half, RadialTaylor &T) {
  const double r = sqrt(s0), p = 1.1283791670955126 * a;
  double En = exp(-a * a * s0), fn = erfc(a * r) / r, gm = 0.0, scale = 1.0;
  for (int n = 0; n < 8; ++n) {
    const double gn = (fn + p * En - gm) / s0;
    T.f[n] = fn * scale;
    T.g[n] = gn * scale;
    fn = -gn / (2.0 * (n + 1));
    En *= -a * a / (n + 1);
    gm = gn;
    scale *= half;
  }
}
__host__ __device__ inline void pair_interval(int i, double R1, double &s0, double &half) {
  const int o = i >> kPtBits, k = i & ((1 << kPtBits) - 1);
  const double lo = ldexp(R1 * R1, -(o + 1));              // S in [2^(62 - o), 2^(63 - o))
  half = ldexp(lo, -(kPtBits + 1));
  s0 = lo + (2 * k + 1) * half;
}
__host__ __device__ inline PairCoef pair_coef(const double *c, const double *minus, double scale) {
  double v[8];
  for (int n = 0; n < 8; ++n) v[n] = scale * (minus ? c[n] - minus[n] : c[n]);
  return PairCoef{v[0], v[1], v[2], v[3], (float)v[4], (float)v[5], (float)v[6], (float)v[7]};
}

__host__ __device__ __forceinline__ int pf_clz(uint64_t v) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}
__host__ __device__ __forceinline__ double pf_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  __builtin_memcpy(&d, &b, 8);
  return d;
#endif
}
__host__ __device__ __forceinline__ float pf_float(uint32_t b) {
#ifdef __CUDA_ARCH__
  return __int_as_float((int)b);
#else
  float f;
  __builtin_memcpy(&f, &b, 4);
  return f;
#endif
}
__host__ __device__ __forceinline__ uint32_t pf_bits(float f) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(f);
#else
  uint32_t b;
  __builtin_memcpy(&b, &f, 4);
  return b;
#endif
}

// v 2^e as a double (truncated to 53 bits), integer instructions only; e + 63 within the normal range
__host__ __device__ __forceinline__ double fix_to_double(int64_t v, int e) {
  const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = pf_clz(a);
  const uint64_t m = a << (z & 63);                        // leading one at bit 63
  // the leading one adds one to the exponent field
  const uint64_t b = ((uint64_t)(uint32_t)(1023 + 62 + e - z) << 52) + (m >> 11);
  return pf_double(a ? sign | b : 0ull);
}
// a normal FP32 value (or zero) as a double, integer instructions only; subnormals give zero
__host__ __device__ __forceinline__ double pf_widen(float f) {
  const uint32_t u = pf_bits(f);
  const uint64_t b = ((uint64_t)(u & 0x80000000u) << 32) | (((uint64_t)(u & 0x7fffffffu) << 29) + (896ull << 52));
  return pf_double((u & 0x7f800000u) ? b : 0ull);
}

// squared distance of the difference d (fractions of W, |d| <= 2^61 per component) as S
__host__ __device__ __forceinline__ uint64_t pair_S(int64_t dx, int64_t dy, int64_t dz) {
  const int32_t xh = (int32_t)(dx >> 31), yh = (int32_t)(dy >> 31), zh = (int32_t)(dz >> 31);
  const int32_t xl = (int32_t)(dx & 0x7fffffff), yl = (int32_t)(dy & 0x7fffffff), zl = (int32_t)(dz & 0x7fffffff);
  const int64_t A = (int64_t)xh * xh + (int64_t)yh * yh + (int64_t)zh * zh;
  const int64_t B = (int64_t)xh * xl + (int64_t)yh * yl + (int64_t)zh * zl;
  const uint64_t C = (uint64_t)((int64_t)xl * xl) + (uint64_t)((int64_t)yl * yl) + (uint64_t)((int64_t)zl * zl);
  // r^2 = A 2^62 + B 2^32 + C in units of (W 2^-64)^2, and R1^2 2^-63 = 2^59 of these units; rounded
  return ((uint64_t)A << 3) + (uint64_t)((B + (int64_t)(C >> 32) + (1ll << 26)) >> 27);
}

struct PairArg {               // where S falls: interval, t, S as a double (units of R1^2)
  int idx;
  double t, s;
  float tf;
};
__host__ __device__ __forceinline__ PairArg pair_arg(uint64_t S) {
  PairArg p;
  const int lz = pf_clz(S);
  const uint64_t M = S << lz;
  p.idx = ((lz - 1) << kPtBits) | (int)((M >> 56) & 127);
  const int64_t tr = (int64_t)(M & ((1ull << 56) - 1)) - (1ll << 55);
  p.t = fix_to_double(tr, -55);
  p.tf = (float)(int32_t)(tr >> 24) * 4.656612873077393e-10f;      // 2^-31
  p.s = pf_double(((uint64_t)(uint32_t)(1023 - lz - 1) << 52) + (M >> 11));   // S 2^-63, truncated
  return p;
}
__host__ __device__ __forceinline__ double pair_poly(const PairCoef &c, const PairArg &p) {
  const float tail = fmaf(p.tf, fmaf(p.tf, fmaf(p.tf, c.c7, c.c6), c.c5), c.c4);
  return fma(p.t, fma(p.t, fma(p.t, fma(p.t, pf_widen(tail), c.c3), c.c2), c.c1), c.c0);
}
// 1 / s for s in [2^-13, 1): FP32 reciprocal, then u (1 + e + e^2) with e = 1 - s u (|e| < 2^-21)
__host__ __device__ __forceinline__ double pair_recip(double s, float sf) {
#ifdef __CUDA_ARCH__
  const float uf = __frcp_rn(sf);
#else
  const float uf = 1.0f / sf;
#endif
  const double u = pf_widen(uf), e = fma(-s, u, 1.0);
  return fma(u, fma(e, e, e), u);
}
// the same value in FP32, without a conversion instruction
__host__ __device__ __forceinline__ float pair_s_float(uint64_t S) {
  const int lz = pf_clz(S);
  return pf_float(((uint32_t)(127 - lz - 1) << 23) + (uint32_t)((S << lz) >> 40));
}

}  // namespace srbe
