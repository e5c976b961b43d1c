// FP64 pair terms on few FP64 instructions (the FP64 form's real-space sums).
//
// GB300 issues 1.7 FP64 FMAs per clock and SM against 64 integer and 128 FP32 operations, so a pair
// written with sqrt, erfc, exp and divisions (about 150 FP64 instructions) costs 90 clocks of an SM.
// Here nearly everything is integer arithmetic, and 7 FP64 FMAs are left (weights and force sums):
//  * coordinates are 64-bit fixed-point fractions of a power-of-two period W >= 8 (rc + margin), so
//    differences (and image shifts) are exact modulo W and every pair within reach has |d| < W / 8 =: R1;
//  * S = r^2 in units of R1^2 2^-63 is formed from 31-bit limbs and rounded once;
//  * S is normalised: its exponent (12 octaves, r >= R1 / 64) and the next 7 bits select an interval, the
//    rest is t in [-1, 1); the radial factor is k0 + t (k1 + ... + t c7): k0..k3 as 64-bit integers with one
//    exponent per interval, the tail in FP32 (its terms are below 2^-30 of 1 / r^3, the scale of a pair's
//    force, so their FP32 rounding is below 2^-53 of it).  The error is bounded on that scale: 5e-16 of
//    1 / r^3 at worst for any alpha r.  Of its own factor a screened pair has less: 2.4e-14 at worst, 2.9e-15 rms,
//    at r = 1.2 nm with alpha 3.5 (plain functions 2.0e-15, 1.0e-15), 2.9e-12 at alpha r = 7.2, where the factor
//    is 3e-22 of 1 / r^3;
//  * 1 / S comes from an FP32 reciprocal and one cubic Newton step, its powers from 64-bit products;
//  * int64 <-> floating-point conversions are assembled with integer instructions.
// A pair closer than R1 / 64 leaves the table and takes the plain FP64 functions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace srbe {

constexpr int kPtOctaves = 12, kPtBits = 7;                // table intervals: 12 octaves of S, 128 each
constexpr int kPtSize = kPtOctaves << kPtBits;
constexpr uint64_t kPtMin = 1ull << (63 - kPtOctaves);     // smallest S of the table

struct __align__(16) PairCoef {                            // radial factor on one interval
  int64_t k0, k1, k2, k3;      // coefficients of (t / 2)^n, Q62 times 2^E
  float c4, c5, c6, c7;        // the same, times 2^-E; the low 12 bits of c7 hold E + 2048
};

// The Taylor expansion (in units of the half interval) of the radial factors around the centre of
// interval i: with s = r^2, f = erfc(a sqrt s) / sqrt s and E = exp(-a^2 s), df/ds = -g / 2 where
// g = (f + (2 a / sqrt pi) E) / s is the force factor -phi'(r) / r, so the Taylor coefficients of f and
// g follow from one another term by term:
//   f_{n+1} = -g_n / (2 (n + 1)),   g_n = (f_n + (2 a / sqrt pi) E_n - g_{n-1}) / s0.
// The interval is 2^-8 of its s on either side, so the first term left out is 2^-64 of c0 from the powers of
// r, and from the exponential x^8 / (256^8 8!) e^-x of 1 / r^3 with x = a^2 s: at most 8e-21 of it (at x = 8),
// although of a strongly screened c0 it is more (1e-15 at x = 17, 2e-13 at x = 35).
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

// v 2^e as a double (rounded), integer instructions only; e + 63 within the normal range
__host__ __device__ __forceinline__ double fix_to_double(int64_t v, int e) {
  const uint64_t sign = (uint64_t)v & 0x8000000000000000ull;
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const int z = pf_clz(a);
  const uint64_t m = a << (z & 63);                        // leading one at bit 63
  // the leading one adds one to the exponent field, and so does a rounding that carries through
  const uint64_t b = ((uint64_t)(uint32_t)(1023 + 62 + e - z) << 52) + (m >> 11) + ((m >> 10) & 1);
  return pf_double(a ? sign | b : 0ull);
}
// f 2^62 as an integer for |f| < 1 (truncated), integer instructions only
__host__ __device__ __forceinline__ int64_t float_to_q62(float f) {
  const uint32_t u = pf_bits(f);
  const int sh = (int)((u >> 23) & 255) - 127 + 39;        // the significand's last bit is worth 2^(e - 23)
  const uint64_t m = (u & 0x7fffffu) | 0x800000u;
  const int64_t v = sh >= 0 ? (int64_t)(m << (sh & 63)) : (sh > -24 ? (int64_t)(m >> (-sh & 63)) : 0);
  return (u >> 31) ? -v : v;
}
// hi 64 bits of a b (signed), without the product of the low halves: within 3 units
__host__ __device__ __forceinline__ int64_t fix_mulhi(int64_t a, int64_t b) {
  const int32_t ah = (int32_t)(a >> 32), bh = (int32_t)(b >> 32);
  const int32_t al = (int32_t)((uint32_t)a >> 1), bl = (int32_t)((uint32_t)b >> 1);   // 31 bits
  return (int64_t)ah * bh + (((int64_t)ah * bl) >> 31) + (((int64_t)bh * al) >> 31);
}

__host__ __device__ inline PairCoef pair_coef(const double *c, const double *minus, double scale) {
  double v[8], top = 0.0;
  for (int n = 0; n < 8; ++n) {
    v[n] = scale * (minus ? c[n] - minus[n] : c[n]) * (double)(1 << n);                  // powers of t / 2
    if (n < 4) top = fmax(top, fabs(v[n]));
  }
  // the exponent that brings the four leading coefficients below 1 (an entry below 1e-280 is zero: its last
  // unit, 2^(E - 62), and any value of the polynomial stay normal doubles)
  int E = 0;
  if (top > 1e-280) frexp(top, &E);
  else for (int n = 0; n < 8; ++n) v[n] = 0.0;
  PairCoef k;
  k.k0 = (int64_t)ldexp(v[0], 62 - E);
  k.k1 = (int64_t)ldexp(v[1], 62 - E);
  k.k2 = (int64_t)ldexp(v[2], 62 - E);
  k.k3 = (int64_t)ldexp(v[3], 62 - E);
  k.c4 = (float)ldexp(v[4], -E);
  k.c5 = (float)ldexp(v[5], -E);
  k.c6 = (float)ldexp(v[6], -E);
  k.c7 = pf_float((pf_bits((float)ldexp(v[7], -E)) & ~4095u) | (uint32_t)(E + 2048));
  return k;
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

struct PairArg {               // where S falls: interval, t / 2 (as Q64 and in FP32), and S normalised
  int idx, lz;
  uint64_t M;                  // S << lz: the significand m in [1, 2) as Q63; S 2^-63 = m 2^-lz
  int64_t t;
  float tf;
};
__host__ __device__ __forceinline__ PairArg pair_arg(uint64_t S) {
  PairArg p;
  p.lz = pf_clz(S);
  p.M = S << p.lz;
  p.idx = ((p.lz - 1) << kPtBits) | (int)((p.M >> 56) & 127);
  p.t = (int64_t)((p.M << 8) ^ (1ull << 63));              // the low 56 bits as a fraction, less 1/2, in Q64
  p.tf = (float)(int32_t)(p.t >> 32) * 2.3283064365386963e-10f;      // 2^-32
  return p;
}
__host__ __device__ __forceinline__ double pair_poly(const PairCoef &c, const PairArg &p) {
  const float tail = fmaf(p.tf, fmaf(p.tf, fmaf(p.tf, c.c7, c.c6), c.c5), c.c4);
  int64_t v = c.k3 + fix_mulhi(p.t, float_to_q62(tail));
  v = c.k2 + fix_mulhi(p.t, v);
  v = c.k1 + fix_mulhi(p.t, v);
  v = c.k0 + fix_mulhi(p.t, v);
  return fix_to_double(v, (int)(pf_bits(c.c7) & 4095) - 2048 - 62);
}
// u^3 and u^4 of u = 1 / (S 2^-63) in integer arithmetic: an FP32 reciprocal u of the significand, then
// u (1 + e + e^2) with e = 1 - m u exact in Q62 (|e| < 2^-21, so the next term is below 2^-63)
__host__ __device__ __forceinline__ void pair_powers(const PairArg &p, double &u3, double &u4) {
  const float mf = pf_float(0x3f800000u + (uint32_t)((p.M << 1) >> 41));        // m, truncated
#ifdef __CUDA_ARCH__
  float uf;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(uf) : "f"(mf));
#else
  const float uf = 1.0f / mf;
#endif
  // uf in (0.5, 1] as Q31: its 24 significand bits below an implicit exponent of -1, or 1.0 itself
  const uint32_t ub = pf_bits(uf);
  const uint32_t U = ub >= 0x3f800000u ? 0x80000000u : ((ub & 0x7fffffu) | 0x800000u) << 7;
  const uint32_t mh = (uint32_t)(p.M >> 32), ml = (uint32_t)p.M;
  const uint64_t prod = (uint64_t)mh * U + (((uint64_t)ml * U) >> 32);          // m u in Q62
  const int64_t e = (int64_t)((1ull << 62) - prod);
  const int32_t eh = (int32_t)(e >> 12);                                        // Q50, |eh| < 2^30
  const int64_t f = e + (((int64_t)eh * eh) >> 38);                             // e + e^2 in Q62
  const int32_t fh = (int32_t)(f >> 12), fl = (int32_t)(f & 4095);
  const int32_t Us = (int32_t)(U >> 1);                                         // Q30 (U's last 7 bits are zero)
  // u in Q62: U Q31 -> Q62, plus u f: Q30 Q50 -> Q62 is >> 18, the low part >> 30
  const int64_t u = ((int64_t)U << 31) + (((int64_t)Us * fh) >> 18) + (((int64_t)Us * fl) >> 30);
  // u in (1/2, 1]: its square as Q60, kept as Q62 for the products
  const int64_t q = fix_mulhi(u, u) << 2;
  u3 = fix_to_double(fix_mulhi(q, u), -60 + 3 * p.lz);
  u4 = fix_to_double(fix_mulhi(q, q), -60 + 4 * p.lz);
}

}  // namespace srbe
