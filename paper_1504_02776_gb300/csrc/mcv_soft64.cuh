// FP64 division, square root and elementary functions on the integer pipes.
//
// GB300 issues FP64 instructions at 1/64 of its FP32 and integer rate (2 lanes per clock per
// SM), so the FP64 kernels are bound by the FP64 pipe while the others idle.  A double's
// division or square root is about 8 to 10 FP64 instructions; on its 53-bit significand it is
// a few 32 x 32 -> 64-bit multiplications: an FP32 seed of 22 bits, one third-order
// (Newton-Schroeder) step in 64-bit fixed point, and the exact remainder where the rounding is
// not yet decided.  The results are those of IEEE round-to-nearest-even, bit for bit;
// operands outside the normal range (zeros, subnormals, infinities, NaN, results that leave
// the normal range) take the FP64 operator.
//
// The functions are compiled once per kernel and called: inlined at their some sixty call
// sites they would make the kernels ten times as large.
//
// exp, log, sin/cos and tan are Taylor series in 64-bit fixed point after the usual argument
// reductions (exp: 2^-n 2^G; log: k ln 2 + 2 atanh((m - 1)/(m + 1)); sin and cos: the nearest
// quarter turn), rounded once to double.  Largest errors in units in the last place of the
// result: at most 0.51 each.
#pragma once

// Measured on a GB300 (cycles per warp instruction and SM sub-partition, throughput): one
// FP64 instruction 64; division 580 -> 130, square root 695 -> 145; the library's exp 1280,
// log 2360, sincos 1790, tan 1950.  With these functions the FP64 powder run (5e6 neutrons)
// went from 9.39 to 5.91 ms, the Bragg powder (2e6) from 4.94 to 3.10 ms, one FP64 run of
// the test cylinder (1e5) from 203 to 115 us.
//
// The header also compiles as plain C++ (the CPU test runs the same arithmetic there).
#include <cmath>
#include <cstdint>
#ifdef __CUDACC__
#include <cuda_runtime.h>
#define MCV_S64 __device__ __forceinline__
#define MCV_S64_CALL static __device__ __noinline__
#else
#include <cstring>
#define MCV_S64 inline
#define MCV_S64_CALL inline
#endif

namespace mcv {
namespace soft64 {

#ifdef __CUDACC__
MCV_S64 uint64_t bits(double x) { return (uint64_t)__double_as_longlong(x); }
MCV_S64 double from_bits(uint64_t b) { return __longlong_as_double((long long)b); }
MCV_S64 float float_of(uint32_t b) { return __uint_as_float(b); }
MCV_S64 uint32_t bits32(float x) { return __float_as_uint(x); }
MCV_S64 uint64_t mul_hi64(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
MCV_S64 uint32_t mul_hi(uint32_t a, uint32_t b) { return __umulhi(a, b); }
MCV_S64 int leading_zeros(uint64_t a) { return __clzll((long long)a); }
// seeds of the reciprocal and of the reciprocal square root: relative error below 2^-22
MCV_S64 float rcp_seed(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
MCV_S64 float rsqrt_seed(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
typedef double2 Pair;
#else
inline uint64_t bits(double x) { uint64_t b; std::memcpy(&b, &x, 8); return b; }
inline double from_bits(uint64_t b) { double x; std::memcpy(&x, &b, 8); return x; }
inline float float_of(uint32_t b) { float x; std::memcpy(&x, &b, 4); return x; }
inline uint32_t bits32(float x) { uint32_t b; std::memcpy(&b, &x, 4); return b; }
inline uint64_t mul_hi64(uint64_t a, uint64_t b) {
  return (uint64_t)(((unsigned __int128)a * b) >> 64);
}
inline uint32_t mul_hi(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
inline int leading_zeros(uint64_t a) { return a ? __builtin_clzll(a) : 64; }
extern int seed_error;  // units in the last place added to the seeds by the test
inline float rcp_seed(float x) { return float_of(bits32(1.0f / x) + (uint32_t)seed_error); }
inline float rsqrt_seed(float x) {
  return float_of(bits32((float)(1.0 / std::sqrt((double)x))) + (uint32_t)seed_error);
}
struct Pair { double x, y; };
#endif

// (a * y) >> 32 for a 64-bit a and a 32-bit y
MCV_S64 uint64_t mul_hi32(uint64_t a, uint32_t y) {
  return (uint64_t)(uint32_t)(a >> 32) * y + (((uint64_t)(uint32_t)a * y) >> 32);
}

// operands outside the ranges of the functions below, out of their way
MCV_S64_CALL double native_div(double a, double b) { return a / b; }
MCV_S64_CALL double native_sqrt(double x) { return ::sqrt(x); }
MCV_S64_CALL double native_exp(double x) { return ::exp(x); }
MCV_S64_CALL double native_log(double x) { return ::log(x); }
MCV_S64_CALL double native_tan(double x) { return ::tan(x); }

// The reciprocal of a divisor, to be used for one or more quotients.
struct Recip {
  double b;       // the divisor
  uint64_t y;     // 2^64 / significand of b (in [1, 2)), error below 2^-61 of 1
};

// 2^64 / b for b in [1, 2) given in units of 2^-63
MCV_S64 uint64_t recip_fixed(uint64_t d) {
  // seed: 1/b in (0.5, 1) from the 24 leading bits, as a fraction of 2^32; the FP32
  // approximation and the truncation leave a relative error below 2^-21.5
  const float fb = float_of(0x3f800000u | ((uint32_t)(d >> 40) & 0x7fffffu));
  const float fy = fminf(fmaxf(rcp_seed(fb), 0.5f), 0x1.fffffep-1f);
  const uint32_t y0 = (bits32(fy) << 8) | 0x80000000u;
  // e = 1 - b y0 in units of 2^-63, then y = y0 (1 + e + e^2): error e^3 < 2^-64
  const int64_t e = (int64_t)(0x8000000000000000ull - mul_hi32(d, y0));
  const int32_t eh = (int32_t)(e >> 14);  // |e| < 2^43
  const int64_t c = e + (int64_t)(((uint64_t)((int64_t)eh * eh)) >> 35);
  const int64_t hi = (int64_t)(int32_t)(c >> 32) * (int64_t)(uint64_t)y0;
  const uint64_t lo = (uint64_t)(uint32_t)c * y0;
  return ((uint64_t)y0 << 32) + ((uint64_t)hi << 1) + (lo >> 31);
}

MCV_S64 Recip recip(double b) {
  const uint64_t mb = (bits(b) & 0xfffffffffffffull) | 0x10000000000000ull;
  return Recip{b, recip_fixed(mb << 11)};
}

// a / r.b, rounded to nearest even
MCV_S64 double div(double a, const Recip& r) {
  const uint64_t A = bits(a), B = bits(r.b);
  const int ea = (int)(A >> 52) & 0x7ff, eb = (int)(B >> 52) & 0x7ff;
  const int e0 = ea - eb + 1023;
  // both normal and the quotient normal whatever its rounding
  if (!((unsigned)(ea - 1) < 2046u && (unsigned)(eb - 1) < 2046u && (unsigned)(e0 - 2) < 2043u))
    return native_div(a, r.b);
  const uint64_t ma = (A & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint64_t mb = (B & 0xfffffffffffffull) | 0x10000000000000ull;
  uint64_t q = mul_hi64(ma << 11, r.y);  // a/b in (0.5, 2) in units of 2^-63, a few units off
  const int up = q >> 63 ? 0 : 1;          // a/b < 1: one bit more
  q <<= up;
  uint64_t m = (q >> 11) + ((unsigned)(q >> 10) & 1u);  // 53 bits, to nearest (or 2^53)
  const unsigned rest = ((unsigned)q - 0x3e0u) & 0x7ffu;
  if (rest < 0x40u) {
    // within 32 units of half a bit: the exact remainder decides (|remainder| < 2^54, so its
    // low 64 bits are enough)
    const int64_t rem = (int64_t)((ma << (52 + up)) - m * mb);
    if (2 * rem > (int64_t)mb) m += 1;
    if (2 * rem < -(int64_t)mb) m -= 1;
  }
  const uint64_t sign = (A ^ B) & 0x8000000000000000ull;
  return from_bits((sign | ((uint64_t)(unsigned)(e0 - up - 1) << 52)) + m);
}

MCV_S64_CALL double div(double a, double b) { return div(a, recip(b)); }
// the same in two calls: the reciprocal's fixed-point significand, then the quotients
MCV_S64_CALL uint64_t recip_of(double b) { return recip(b).y; }
MCV_S64_CALL double div_by(double a, double b, uint64_t y) { return div(a, Recip{b, y}); }

// sqrt(x), rounded to nearest even
MCV_S64_CALL double sqrt(double x) {
  const uint64_t X = bits(x);
  const int e = (int)(X >> 52);  // with the sign bit: negative numbers leave the range below
  if (!((unsigned)(e - 1) < 2046u)) return native_sqrt(x);
  const uint64_t mx = (X & 0xfffffffffffffull) | 0x10000000000000ull;
  const int odd = (e & 1) ? 0 : 1;             // unbiased exponent odd: significand in [2, 4)
  const uint64_t v = mx << (10 + odd);         // in [1, 4), units of 2^-62
  // seed 1/sqrt(v) in (0.5, 1) from the 24 leading bits, as a fraction of 2^32
  const float fv = float_of((0x3f800000u + ((unsigned)odd << 23)) |
                                   ((uint32_t)(mx >> 29) & 0x7fffffu));
  const float fy = fminf(fmaxf(rsqrt_seed(fv), 0.5f), 0x1.fffffep-1f);
  const uint32_t y = (bits32(fy) << 8) | 0x80000000u;
  // e = 1 - v y^2 in units of 2^-62; sqrt(v) = v y (1 + e/2 + 3 e^2/8), error e^3 < 2^-62
  const int64_t er = (int64_t)(0x4000000000000000ull - mul_hi64(v, (uint64_t)y * y));
  const int32_t eh = (int32_t)(er >> 13);      // |er| < 2^43
  const int64_t c = (er >> 1) + (int64_t)((3ull * (uint64_t)((int64_t)eh * eh)) >> 39);
  const uint64_t h = mul_hi32(v, y);           // v y in [1, 2), units of 2^-62
  // h c / 2^62: c scaled by 2^20 keeps the product's high word exact to a unit
  const int64_t cs = c << 20;
  int64_t hc = (int64_t)mul_hi64(h, (uint64_t)cs);
  if (cs < 0) hc -= (int64_t)h;
  const uint64_t s = h + (uint64_t)(hc >> 18);
  uint64_t m = (s + 0x200u) >> 10;             // 53 bits, to nearest
  const unsigned rest = ((unsigned)s - 0x1e0u) & 0x3ffu;
  if (rest < 0x40u) {
    // the exact remainder v 2^104 - m^2 decides (its low 64 bits: |remainder| <= 2^54)
    const int64_t rem = (int64_t)((mx << (52 + odd)) - m * m);
    if (rem > (int64_t)m) m += 1;
    if (rem <= -(int64_t)m) m -= 1;
  }
  const unsigned er2 = (unsigned)((e + 1023) >> 1);
  return from_bits(((uint64_t)(er2 - 1) << 52) + m);
}

// v 2^(ex - 63) for a v with its top bit set, rounded to nearest
MCV_S64 double pack(uint64_t sign, uint64_t v, int ex) {
  return from_bits(sign + ((uint64_t)(unsigned)(ex + 1022) << 52) + (v >> 11) +
                   ((unsigned)(v >> 10) & 1u));
}

// sin (x) and cos (y) of fl(2 pi u), u in (0, 1].  The argument is reduced with 128 bits of 2/pi
// and the reduced argument keeps its own exponent, so both are relatively accurate however near
// a quarter turn they are (a double in (0, 2 pi) is at least 2^-60 away from one).
MCV_S64_CALL Pair sincos2pi(double u) {
  const uint64_t A = bits(6.283185307179586 * u);
  const int e = (int)(A >> 52) - 1023;  // -54 .. 2
  const uint64_t v = ((A & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
  // x in quarter turns: x 2/pi = (hi, lo) 2^(e - 127)
  uint64_t lo = v * 0xa2f9836e4e441529ull;
  uint64_t hi = mul_hi64(v, 0xa2f9836e4e441529ull);
  const uint64_t low = mul_hi64(v, 0xfc2757d1f534ddc0ull);
  lo += low;
  hi += lo < low ? 1 : 0;
  // the nearest whole number of them, and the distance to it: (hi, lo) 2^(-128 - drop)
  unsigned quad = 0;
  int drop = 0;
  if (e >= -1) {
    const int sh = e + 1;
    if (sh) {
      quad = (unsigned)(hi >> (64 - sh));
      hi = (hi << sh) | (lo >> (64 - sh));
      lo <<= sh;
    }
  } else {
    drop = -1 - e;
  }
  const uint64_t neg = drop == 0 ? hi & 0x8000000000000000ull : 0;
  if (neg) {
    quad += 1;
    lo = 0ull - lo;
    hi = ~hi + (lo == 0 ? 1 : 0);
  }
  // an 2^(-64 - la): its leading 64 bits
  if (hi == 0) {
    hi = lo;
    lo = 0;
    drop += 64;
  }
  const int lh = leading_zeros(hi | 1);
  const uint64_t an = lh ? (hi << lh) | (lo >> (64 - lh)) : hi;
  const int la = lh + drop;
  const uint64_t a = la < 64 ? an >> la : 0;  // quarter turns, at most 1/2, units of 2^-64
  const uint64_t w = mul_hi64(a, a);
  const uint32_t w32 = (uint32_t)(w >> 32);
  // sin(pi/2 a) = a S(w), cos(pi/2 a) = C(w): Taylor coefficients (pi/2)^n / n!, units of 2^-63
  uint64_t S = 0x355d865ull;
  S = 0x16fadb9f1ull - mul_hi32(S, w32);
  S = 0x7a3d0d3406ull - mul_hi32(S, w32);
  S = 0x1e3074fde887ull - mul_hi32(S, w32);
  S = 0x541e0d21fb9e0ull - mul_hi64(S, w);
  S = 0x9969667315ec2eull - mul_hi64(S, w);
  S = 0xa335e33bad570e9ull - mul_hi64(S, w);
  S = 0x52aef39896f94afbull - mul_hi64(S, w);
  S = 0xc90fdaa22168c235ull - mul_hi64(S, w);
  uint64_t C = 0x4a8316ull;
  C = 0x2418c586ull - mul_hi32(C, w32);
  C = 0xdb7127a26ull - mul_hi32(C, w32);
  C = 0x3f3a7146ec8ull - mul_hi32(C, w32);
  C = 0xd368f9510254ull - mul_hi32(C, w32);
  C = 0x1e1f506891babbull - mul_hi64(C, w);
  C = 0x2aba78fc797ff40ull - mul_hi64(C, w);
  C = 0x20783e1036b58767ull - mul_hi64(C, w);
  C = 0x9de9e64df22ef2d2ull - mul_hi64(C, w);
  C = 0x8000000000000000ull - mul_hi64(C, w);
  const uint64_t p = mul_hi64(an, S);  // at least 2^62
  const int lp = leading_zeros((p | 1));
  double s = pack(0, p << lp, -la - lp);
  const int lc = leading_zeros(C);
  double c = pack(0, C << lc, -lc);
  s = from_bits(bits(s) ^ neg);
  const bool odd = quad & 1;
  const uint64_t vs = bits(odd ? c : s), vc = bits(odd ? s : c);
  return Pair{from_bits(vs ^ ((uint64_t)(quad & 2) << 62)),
                      from_bits(vc ^ ((uint64_t)((quad + 1) & 2) << 62))};
}

// exp(x); -700 <= x <= 0 in fixed point, other arguments by the library
MCV_S64_CALL double exp(double x) {
  const uint64_t A = bits(x);
  if (!(A >= 0x8000000000000000ull && A <= 0xc085e00000000000ull)) return native_exp(x);
  const int e = ((int)(A >> 52) & 0x7ff) - 1023;
  if (e < -54) return 1.0;
  const uint64_t mx = (A & 0xfffffffffffffull) | 0x10000000000000ull;
  // |x| log2(e) = k + F = (hi, lo) 2^(e - 126), F in units of 2^-64; the 32 bits of log2(e) behind
  // the first 64 count once |x| is large
  const uint64_t v = mx << 11;
  const uint64_t low = mul_hi32(v, 0xbe87fed0u);
  const uint64_t lo = v * 0xb8aa3b295c17f0bbull + low;
  const uint64_t hi = mul_hi64(v, 0xb8aa3b295c17f0bbull) + (lo < low ? 1 : 0);
  const int k = e >= -1 ? (int)(hi >> (62 - e)) : 0;
  const uint64_t F = e >= -1 ? (hi << (e + 2)) | (lo >> (62 - e)) : hi >> (-e - 2);
  const uint64_t G = 0ull - F;       // 2^-(k + F) = 2^-(k + 1) 2^(1 - F)
  const int n = F ? k + 1 : k;
  const uint32_t g32 = (uint32_t)(G >> 32);
  // 2^G = 1 + G t: Taylor coefficients ln(2)^n / n!, the small ones in 32 bits
  uint32_t c = 16u;
  c = 408u + mul_hi(c, g32);
  c = 10013u + mul_hi(c, g32);
  c = 231133u + mul_hi(c, g32);
  c = 5001817u + mul_hi(c, g32);
  c = 101025356u + mul_hi(c, g32);
  c = 1894734148u + mul_hi(c, g32);
  uint64_t t = c >> 3;
  t = 0xf465639bull + mul_hi64(t, G);
  t = 0xf267a8ac6ull + mul_hi64(t, G);
  t = 0xda929e9cafull + mul_hi64(t, G);
  t = 0xb160111d2e4ull + mul_hi64(t, G);
  t = 0x7ff2ff1622c3ull + mul_hi64(t, G);
  t = 0x50c244be1b1e2ull + mul_hi64(t, G);
  t = 0x2bb0ffcf14ce62ull + mul_hi64(t, G);
  t = 0x13b2ab6fba4e773ull + mul_hi64(t, G);
  t = 0x71ac235c1282fe3ull + mul_hi64(t, G);
  t = 0x1ebfbdff82c58ea8ull + mul_hi64(t, G);
  t = 0x58b90bfbe8e7bcd6ull + mul_hi64(t, G);
  t = mul_hi64(t, G);
  return from_bits(((uint64_t)(unsigned)(1023 - n) << 52) + ((t + 0x400u) >> 11));
}

// log(x) for normal x within 2^-63 .. 2^63, other arguments by the library
MCV_S64_CALL double log(double x) {
  const uint64_t A = bits(x);
  const int e = (int)(A >> 52) - 1023;
  if (!((unsigned)(e + 62) < 124u)) return native_log(x);
  const uint64_t mx = (A & 0xfffffffffffffull) | 0x10000000000000ull;
  // x = 2^k m with m in (0.707, 1.414): significands above sqrt(2) are halved
  const bool half = mx > 0x16a09e667f3bcdull;
  const int k = e + (half ? 1 : 0);
  const uint64_t z = half ? 0x20000000000000ull - mx : mx - 0x10000000000000ull;
  const uint64_t d = (mx + (half ? 0x20000000000000ull : 0x10000000000000ull)) << 10;
  // |f| = |m - 1| / (m + 1) = fn 2^(-lz - 53)
  const int lz = leading_zeros((z | 1));
  const uint64_t fn = mul_hi64(z << lz, recip_fixed(d));
  const uint64_t f = lz >= 13 ? fn >> (lz - 13) : fn << 1;  // units of 2^-66
  const uint64_t w = mul_hi64(f, f);                      // f^2, units of 2^-68
  const uint32_t w32 = (uint32_t)(w >> 32);
  // atanh(f) = f T, T = sum f^2n / (2n + 1), the small terms in 32 bits
  uint32_t c = 0xa3d70a4u;                                  // 1/25, units of 2^-32
  c = 0xb21642du + (mul_hi(c, w32) >> 4);
  c = 0xc30c30cu + (mul_hi(c, w32) >> 4);
  c = 0xd79435eu + (mul_hi(c, w32) >> 4);
  c = 0xf0f0f0fu + (mul_hi(c, w32) >> 4);
  c = 0x11111111u + (mul_hi(c, w32) >> 4);
  c = 0x13b13b14u + (mul_hi(c, w32) >> 4);
  uint64_t t = (uint64_t)c << 31;
  t = 0xba2e8ba2e8ba2e9ull + (mul_hi64(t, w) >> 4);
  t = 0xe38e38e38e38e39ull + (mul_hi64(t, w) >> 4);
  t = 0x1249249249249249ull + (mul_hi64(t, w) >> 4);
  t = 0x199999999999999aull + (mul_hi64(t, w) >> 4);
  t = 0x2aaaaaaaaaaaaaabull + (mul_hi64(t, w) >> 4);
  t = 0x8000000000000000ull + (mul_hi64(t, w) >> 4);
  const uint64_t p = z ? mul_hi64(fn, t) : 0;             // |log m| = p 2^(-lz - 51)
  if (k == 0) {
    if (p == 0) return 0.0;
    const int l = leading_zeros(p);
    return pack(half ? 0x8000000000000000ull : 0, p << l, 12 - l - lz);
  }
  // |k| ln 2 +- |log m| in 128 bits, units of 2^-122: a unit of the leading word alone is a
  // sixteenth of the last place of a result below 1
  const uint64_t ka = (uint64_t)(unsigned)(k < 0 ? -k : k);
  const uint64_t big = ka * 0x2c5c85fdf473de6ull + mul_hi64(ka, 0xaf278ece600fcbdaull);
  const uint64_t big_lo = ka * 0xaf278ece600fcbdaull;
  const int sh = lz - 7;  // 5 or more
  const uint64_t small = p >> sh, small_lo = p << (64 - sh);
  uint64_t mag, mag_lo;
  if ((k < 0) == half) {
    mag_lo = big_lo + small_lo;
    mag = big + small + (mag_lo < big_lo ? 1 : 0);
  } else {
    mag_lo = big_lo - small_lo;
    mag = big - small - (big_lo < small_lo ? 1 : 0);
  }
  const int l = leading_zeros(mag);
  return pack(k < 0 ? 0x8000000000000000ull : 0, (mag << l) | (mag_lo >> 1 >> (63 - l)), 5 - l);
}

// tan(x); 2^-60 < |x| < 2^-4 in fixed point, other arguments by the library
MCV_S64_CALL double tan(double x) {
  const uint64_t A = bits(x);
  const int e = ((int)(A >> 52) & 0x7ff) - 1023;
  if (!((unsigned)(e + 60) < 56u)) return native_tan(x);
  const uint64_t v = ((A & 0xfffffffffffffull) | 0x10000000000000ull) << 11;
  const uint64_t f = v >> (-e - 1);                         // |x| < 2^-4, units of 2^-64
  const uint64_t w = mul_hi64(f, f);
  const uint32_t w32 = (uint32_t)(w >> 32);
  // tan(x) = x + x^3 T(x^2)
  uint64_t t = 0x5f68d914add78bull;
  t = 0xeb69e870abeefeull + mul_hi32(t, w32);
  t = 0x244dc6abcd84792ull + mul_hi32(t, w32);
  t = 0x5993d220b043e7dull + mul_hi32(t, w32);
  t = 0xdd0dd0dd0dd0dd1ull + mul_hi64(t, w);
  t = 0x2222222222222222ull + mul_hi64(t, w);
  t = 0x5555555555555555ull + mul_hi64(t, w);
  // v (1 + x^2 T), x^2 T < 2^-9
  const uint64_t q = (v >> 1) + (mul_hi64(v, mul_hi64(t, w)) >> 1);  // in [2^62, 2^63.01)
  const int l = leading_zeros(q);
  return pack(A & 0x8000000000000000ull, q << l, e + 1 - l);
}

// ---- tests and conversions (an FP64 comparison or conversion costs what an FP64 addition does,
// 64 cycles; these are 2 to 15 integer instructions.  General comparisons, with NaN and signed
// zeros some 20 instructions each, were slower inlined than the FP64 pipe's: code size) ------
MCV_S64 bool is_zero(double x) { return (bits(x) << 1) == 0; }
// a < b for a, b >= 0 that are not NaN
MCV_S64 bool lt_nonneg(double a, double b) { return (int64_t)bits(a) < (int64_t)bits(b); }
MCV_S64 bool positive(double x) {
  const int64_t b = (int64_t)bits(x);
  return b > 0 && b <= 0x7ff0000000000000ll;
}
// floor(x) where 0 <= x < n (n < 2^31), else -1
MCV_S64 int index_below(double x, int n) {
  const uint64_t b = bits(x);
  const int e = (int)(b >> 52);
  if (e < 1023 || b == 0x8000000000000000ull) return n > 0 ? 0 : -1;
  if (e >= 1023 + 31) return -1;  // too large, negative (the sign bit) or NaN
  const uint32_t m = (uint32_t)(((b & 0xfffffffffffffull) | 0x10000000000000ull) >> (1075 - e));
  return m < (uint32_t)n ? (int)m : -1;
}
// floor(x) clamped to 0 .. n - 1 (NaN: 0)
MCV_S64 int index_clamped(double x, int n) {
  const uint64_t b = bits(x);
  const int e = (int)(b >> 52);
  if (e < 1023 || e > 2047 || b > 0x7ff0000000000000ull) return 0;
  if (e >= 1023 + 31) return n - 1;
  const uint32_t m = (uint32_t)(((b & 0xfffffffffffffull) | 0x10000000000000ull) >> (1075 - e));
  return m < (uint32_t)n ? (int)m : n - 1;
}
// (2 k + 1) 2^-54 for the 53 bits k = hi 2^21 + (lo >> 11), rounded to nearest even
MCV_S64 double uniform53(uint32_t hi, uint32_t lo) {
  const uint64_t m = ((uint64_t)hi << 22) | (lo >> 10) | 1u;
  const int lz = leading_zeros(m);  // 10 or more: only 54-bit values round, and those are ties
  const uint64_t v = m << lz;
  const uint64_t q = v >> 11;
  return from_bits(((uint64_t)(unsigned)(1031 - lz) << 52) + q + ((v >> 10) & q & 1u));
}

}  // namespace soft64
}  // namespace mcv
