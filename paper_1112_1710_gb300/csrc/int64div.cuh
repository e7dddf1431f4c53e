// int64div.cuh -- FP64 division and square root, correctly rounded, on the
// integer and FP32 pipes, and FP64 sign tests and scalings on the integer pipe.
//
// GB300 issues one FP64 warp instruction per SM every 16 cycles (2 lanes per
// clock) but two integer warp instructions per cycle, and the FP64 stages of
// the advance keep the FP64 pipe 82-89% busy while 7-8% of the issue slots
// are used.  A division on the FP64 pipe is about nine of its instructions
// (some 140 cycles of an SM); the same quotient by long division in integers
// is about 60 integer instructions (some 30 cycles of a pipe that idles).
//
// Division: the schoolbook long division with estimated quotient digits
// (Knuth, The Art of Computer Programming, vol. 2, Sec. 4.3.1), two digits of
// 27 bits, each estimated from below with a 31-bit reciprocal of the divisor's
// leading bits (an FP32 reciprocal refined by one Newton step in fixed point);
// the exact remainder then settles the last unit, so the 54-bit quotient is
// its floor and the rounding to 53 bits is exact.  A quotient of two 53-bit
// significands is never halfway between two of them (the odd 54-bit quotient
// times the divisor would have to be a multiple of 2^53), so round to nearest
// is (q + 1) >> 1.  Square root: the same with digits of the root, which is
// never halfway either.  Both give the bits of IEEE division and square root;
// operands or results outside the normal range take the hardware operation.
//
// Measured on GB300 (128^3 blast, per launch, with the selected-side HLLD of
// physics.cuh): contracted k_flux 3.43 -> 1.54 ms and k_pred 2.53 -> 1.97 ms;
// parity build, 90 x 75 x 66: k_flux 1.39 -> 0.63 ms, k_pred 0.98 -> 0.65 ms.
#pragma once

#include <cstdint>
#include <cstring>

#ifdef __CUDACC__
#define MHD_HD __host__ __device__ __forceinline__
#else
#define MHD_HD inline
#endif

namespace mhd {
namespace i64 {

MHD_HD uint64_t bits(double x) {
#ifdef __CUDA_ARCH__
  return (uint64_t)__double_as_longlong(x);
#else
  uint64_t u;
  std::memcpy(&u, &x, 8);
  return u;
#endif
}
MHD_HD double value(uint64_t u) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)u);
#else
  double x;
  std::memcpy(&x, &u, 8);
  return x;
#endif
}
MHD_HD uint32_t fbits(float x) {
#ifdef __CUDA_ARCH__
  return __float_as_uint(x);
#else
  uint32_t u;
  std::memcpy(&u, &x, 4);
  return u;
#endif
}
MHD_HD float fvalue(uint32_t u) {
#ifdef __CUDA_ARCH__
  return __uint_as_float(u);
#else
  float x;
  std::memcpy(&x, &u, 4);
  return x;
#endif
}
MHD_HD uint32_t mulhi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }

// FP32 seeds: 1/f and 1/sqrt(f); any value within 2^-22 relative will do
#ifdef __CUDA_ARCH__
MHD_HD float seed_rcp(float f) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  return r;
}
MHD_HD float seed_rsqrt(float f) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(f));
  return r;
}
#else
extern float (*seed_rcp)(float);    // the host test's stand-ins
extern float (*seed_rsqrt)(float);
#endif

// A seed g in (1/2, 1] as a fraction of 31 bits, lowered by 1.25 2^-21 so that
// the seed's error (2^-22), the operand's truncation (2^-23) and the rounding
// here (2^-23) leave it below the true value: the significand of 1 + g.
MHD_HD uint32_t fraction31(float g) {
#ifdef __CUDA_ARCH__
  const float h = __fmaf_rn(g, 0.9999994f, 1.0f);
#else
  const float h = __builtin_fmaf(g, 0.9999994f, 1.0f);
#endif
  return (fbits(h) << 9) >> 1;
}

// floor(2^32 / D) within a few units, from below, D = dn / 2^31 in [1, 2) (and
// the bits of D below dn's last counted as one)
MHD_HD uint32_t reciprocal(uint32_t dn) {
  const uint32_t y0 = fraction31(seed_rcp(fvalue(0x3f800000u | ((dn >> 8) & 0x7fffffu))));
  const uint64_t p = (uint64_t)y0 * dn + y0;        // 2^62 (1 - e), 0 < e < 2^-19
  const uint32_t e = (uint32_t)((~p) >> 11);        // e 2^51
  return (y0 << 1) + (mulhi(y0, e) >> 18);
}

constexpr uint32_t kHidden = 0x100000u;

// a * 2^K / b (K = 0 or 1) rounded to nearest.
template <int K> MHD_HD double div_scaled(double a, double b) {
  const uint64_t ua = bits(a), ub = bits(b);
  const uint32_t ah = (uint32_t)(ua >> 32), bh = (uint32_t)(ub >> 32);
  const uint32_t ea = (ah >> 20) & 0x7ffu, eb = (bh >> 20) & 0x7ffu;
  const uint64_t ma = ((uint64_t)((ah & 0xfffffu) | kHidden) << 32) | (uint32_t)ua;
  const uint64_t mb = ((uint64_t)((bh & 0xfffffu) | kHidden) << 32) | (uint32_t)ub;
  const int s = ma < mb ? 1 : 0;
  const int er = (int)ea - (int)eb + 1022 + K - s;  // exponent field of the result less one
  const uint32_t sign = (ah ^ bh) & 0x80000000u;
  const bool ok = ea - 1u < 0x7feu - K && eb - 1u < 0x7feu && (uint32_t)er < 0x7fdu;
  const bool zero = (ua << 1) == 0 && eb - 1u < 0x7feu;  // +-0 / normal
  if (!ok && !zero) return K ? (a + a) / b : a / b;
  const uint32_t y = reciprocal((uint32_t)(mb >> 21));
  const uint64_t n = ma << s;                       // n / mb in [1, 2)
  const uint32_t q1 = mulhi((uint32_t)(n >> 22), y) >> 4;
  const uint64_t r1 = (n << 26) - (uint64_t)q1 * mb;
  const uint32_t q2 = mulhi((uint32_t)(r1 >> 23), y) >> 2;
  const uint64_t r2 = (r1 << 27) - (uint64_t)q2 * mb;
  uint64_t q = ((uint64_t)q1 << 27) + q2;
  q += (r2 >= mb ? 2u : 1u);                        // the floor, plus one to round
  if (r2 >= 2 * mb) q += 1;
  const uint64_t m = q >> 1;
  const uint32_t hi = (uint32_t)(m >> 32) + ((uint32_t)er << 20) + sign;
  return value(ok ? ((uint64_t)hi << 32) | (uint32_t)m : (uint64_t)sign << 32);
}

MHD_HD double div(double a, double b) { return div_scaled<0>(a, b); }

// sqrt(a) rounded to nearest.
MHD_HD double sqrt_rn(double a) {
  const uint64_t ua = bits(a);
  const uint32_t ah = (uint32_t)(ua >> 32);
  const uint32_t ea = ah >> 20;
  const bool ok = ea - 1u < 0x7feu;                 // positive and normal
  if (!ok) {
#ifdef __CUDA_ARCH__
    return __dsqrt_rn(a);
#else
    return __builtin_sqrt(a);
#endif
  }
  const uint32_t odd = (ea & 1u) ^ 1u;              // odd power of two (1023 is even)
  const uint64_t m = (((uint64_t)((ah & 0xfffffu) | kHidden) << 32) | (uint32_t)ua) << odd;  // v 2^52, v in [1, 4)
  const uint32_t v = (uint32_t)(m >> 22);           // v 2^30
  // the seed of 1/sqrt(v) in (1/2, 1], refined: y 2^32
  const float f = fvalue(((127u + odd) << 23) | ((uint32_t)(ua >> 29) & 0x7fffffu));
  const uint32_t y0 = fraction31(seed_rsqrt(f));
  const uint32_t t = mulhi(y0 << 1, y0 << 1);       // y0^2 2^32
  const uint64_t p = (uint64_t)t * v + t;           // 2^62 (1 - e), 0 < e < 2^-18
  const uint32_t e = (uint32_t)((~p) >> 12);        // e 2^50
  const uint32_t y = (y0 << 1) + (mulhi(y0, e) >> 18);
  // the root in two digits: s1 to nearest, then t2 from the exact remainder
  const uint32_t s1 = (mulhi(v, y) + 8u) >> 4;
  const int32_t r1 = (int32_t)(uint32_t)(m - (uint64_t)s1 * s1);
  const int32_t t2 = (int32_t)(((int64_t)r1 * y) >> 32) - 2;
  const uint64_t s = ((uint64_t)s1 << 27) + (uint64_t)(int64_t)t2;
  const uint64_t r = ((uint64_t)(uint32_t)r1 << 54) - (uint64_t)(int64_t)t2 * (((uint64_t)s1 << 28) + (uint64_t)(int64_t)t2);
  uint64_t q = s + 1;
  if (r > 2 * s) q += 1;                            // (s + 1)^2 - s^2 = 2 s + 1
  if (r >= 4 * s + 4) q += 1;
  if (r >= 6 * s + 9) q += 1;
  const uint64_t w = q >> 1;
  const uint32_t er = ((ea - 1u) >> 1) + 511u;  // exponent field of the result less one
  return value(w + ((uint64_t)er << 52));
}

// x * 2^K, |K| <= 2, the exponent field moved; in integers throughout (a
// branch to an FP64 multiplication would be turned into a predicated one,
// which takes the FP64 pipe's time all the same).
template <int K> MHD_HD double scale(double x) {
  const uint64_t u = bits(x);
  const uint32_t h = (uint32_t)(u >> 32), e = (h >> 20) & 0x7ffu;
  constexpr uint32_t least = K < 0 ? 1 - K : 1, most = K < 0 ? 0x7fe : 0x7fe - K;
  if (e - least <= most - least) return value(((uint64_t)(h + ((uint32_t)K << 20)) << 32) | (uint32_t)u);
  if (e == 0x7ffu || (u << 1) == 0) return x;
  const uint64_t s = u & 0x8000000000000000ull;
  if (K > 0) {  // overflow, or a subnormal doubled (the carry is the exponent)
    if (e != 0) return value(s | 0x7ff0000000000000ull);
    const double y = value(s | ((u & 0xfffffffffffffull) << 1));
    return K > 1 ? scale<(K > 1 ? K - 1 : 1)>(y) : y;
  }
  // subnormal result: the significand shifted right, rounded to even
  const uint64_t f = u & 0xfffffffffffffull, m = e ? f | 0x10000000000000ull : f;
  constexpr int k = K < 0 ? -K : 1;
  const int down = k - (e > 1u ? (int)e - 1 : 0);
  uint64_t r = m >> down;
  const uint64_t rest = m - (r << down), half = 1ull << (down - 1);
  if (rest > half || (rest == half && (r & 1))) r += 1;
  return value(s | r);
}

// The double equal to x, in integers (a conversion instruction takes the FP64
// pipe's time).
MHD_HD double widen(float x) {
  const uint32_t f = fbits(x), m = f & 0x7fffffu, e = (f >> 23) & 0xffu, sign = f & 0x80000000u;
  if (e - 1u < 0xfeu) return value(((uint64_t)(sign | (((f & 0x7fffffffu) >> 3) + (896u << 20))) << 32) | (uint64_t)(f << 29));
  if (e == 0xffu) return value(((uint64_t)(sign | 0x7ff00000u | (m >> 3)) << 32) | (uint64_t)(m << 29));
  if (m == 0) return value((uint64_t)sign << 32);
  int k = 0;  // subnormal: the leading bit to position 23
  uint32_t n = m;
  while (!(n & 0x800000u)) n <<= 1, ++k;
  return value(((uint64_t)(sign | ((uint32_t)(897 - k) << 20) | ((n & 0x7fffffu) >> 3)) << 32) | (uint64_t)(n << 29));
}

// x > 0, x < 0, x >= 0 (all false for NaN)
MHD_HD bool pos(double x) { return bits(x) - 1u < 0x7ff0000000000000ull; }
MHD_HD bool neg(double x) { return bits(x) - 0x8000000000000001ull < 0x7ff0000000000000ull; }
MHD_HD bool ge0(double x) { return bits(x) <= 0x7ff0000000000000ull || bits(x) == 0x8000000000000000ull; }
// |x| > t for t >= 0, not NaN
MHD_HD bool abs_gt(double x, double t) {
  const uint64_t m = bits(x) & 0x7fffffffffffffffull;
  return m > (bits(t) & 0x7fffffffffffffffull) && m <= 0x7ff0000000000000ull;
}
// a < b for a, b >= 0, not NaN
MHD_HD bool less_mag(double a, double b) {
  return (bits(a) & 0x7fffffffffffffffull) < (bits(b) & 0x7fffffffffffffffull);
}
MHD_HD bool nan(double x) { return (bits(x) & 0x7fffffffffffffffull) > 0x7ff0000000000000ull; }
// any of the three an infinity or NaN?  (their upper words' exponents)
MHD_HD bool any_special(double a, double b, double c) {
  const uint32_t x = (uint32_t)(bits(a) >> 32) << 1, y = (uint32_t)(bits(b) >> 32) << 1, z = (uint32_t)(bits(c) >> 32) << 1;
  const uint32_t m = x > y ? x : y;
  return (m > z ? m : z) >= 0xffe00000u;
}
MHD_HD bool special(double a) { return (uint32_t)(bits(a) >> 32) << 1 >= 0xffe00000u; }
// Is |d| > 1e-12 max(a1 a2, b) plain from the exponents (b finite)?
MHD_HD bool clearly_above(double d, double a1, double a2, double b) {
  const int ed = (int)(bits(d) >> 52) & 0x7ff, e1 = (int)(bits(a1) >> 52) & 0x7ff,
            e2 = (int)(bits(a2) >> 52) & 0x7ff, eb = (int)(bits(b) >> 52) & 0x7ff;
  const int ea = e1 + e2 - 1022;  // a1 a2 < 2^(ea + 1 - 1023)
  const int m = ea > eb ? ea : eb;
  return ed != 0 && e1 < 0x7ff && e2 < 0x7ff && eb < 0x7ff && ed + 38 > m;
}

}  // namespace i64
}  // namespace mhd
