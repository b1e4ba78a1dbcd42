// FP64 reciprocal, quotient, square roots and powers of positive arguments computed
// in 64-bit fixed point on the integer pipe.
//
// GB300's FP64 unit takes a warp's instruction in 64 cycles on each of an SM's
// four partitions, whatever its lanes, where an integer instruction takes 2: a
// 64 x 64-bit product's upper half (about eight instructions) is several times
// cheaper than one FP64 multiply-add, and a division, square root or power is
// some 10, 10 and 26 of those.  The operands' significands become 64-bit fixed-point
// numbers (Qn: n fractional bits), and the arithmetic below keeps about 60 bits.
// Reciprocal, quotient and square root are then rounded by their exact remainders, so
// they are the bits of the divisions and roots of IEEE 754; x^(-1/2) and x^a are rounded
// from the 60 bits, to at most 0.52 and 0.59 ulp (CUDA documents 1 and 1).
// Every value is the same in every kernel that inlines these.  Arguments outside
// the ranges stated (zero, negative, infinite, NaN, extreme exponents) go to
// CUDA's own functions.
#pragma once

#include <cuda_runtime.h>

#include "pow64_tables.cuh"

namespace amm {

using u64 = unsigned long long;
using i64 = long long;

__device__ __forceinline__ float approx_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float approx_rsqrt(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

static __device__ __noinline__ double div64_rare(double a, double b) { return a / b; }
static __device__ __noinline__ double sqrt64_rare(double x) { return sqrt(x); }
static __device__ __noinline__ double rsqrt64_rare(double x) { return rsqrt(x); }
static __device__ __noinline__ double pow64_rare(double x, double a) { return pow(x, a); }

__device__ __forceinline__ u64 significand(double x) {
  return ((u64)__double_as_longlong(x) & 0xfffffffffffffull) | 0x10000000000000ull;
}
// y0 (1 + t): y0 in (1/2, 1] from the FP32 approximation, t in Q63, |t| < 2^-21; Q61
__device__ __forceinline__ u64 refine(unsigned y0, i64 t) {
  const i64 z = (i64)((u64)y0 * (unsigned)t >> 32) + (i64)(int)y0 * (int)(t >> 32);
  return ((u64)y0 << 31) + (u64)z;
}

// 1/m for a significand m (Q52), in (1/2, 1], Q61.  With e = 1 - m y0 (|e| < 2^-21),
// 1/m = y0 (1 + e + e^2 + ...), the next term below 2^-63.
__device__ __forceinline__ u64 recip_q61(u64 m) {
  const float f = __uint_as_float(0x3f800000u | ((unsigned)(m >> 29) & 0x7fffffu));
  const unsigned y0 = (unsigned)(approx_rcp(f) * 1073741824.0f);           // Q30, exact
  const u64 x = m << 11;                                                    // Q63
  const u64 p = (x >> 32) * y0 + ((x & 0xffffffffu) * y0 >> 32);            // m y0, Q61
  const i64 e = (i64)((1ull << 61) - p);
  const int s = (int)(e >> 9);                                              // Q52
  return refine(y0, (e << 2) + ((i64)s * s >> 41));
}

// m^(-1/2) for m in [1, 4), Q62, in (1/2, 1], Q61.  With e = 1 - m y0^2, m^(-1/2) =
// y0 (1 + e/2 + 3 e^2/8 + ...).  f: m in FP32 (truncated).
__device__ __forceinline__ u64 rsqrt_q61(u64 m, float f) {
  const unsigned y0 = (unsigned)(approx_rsqrt(f) * 1073741824.0f);         // Q30
  const u64 p = __umul64hi(m, (u64)y0 * y0 << 3);                           // m y0^2, Q61
  const i64 e = (i64)((1ull << 61) - p);
  const int s = (int)(e >> 9);                                              // Q52
  return refine(y0, (e << 1) + (i64)((u64)((i64)s * s) * 3 >> 44));
}

__device__ __forceinline__ unsigned exponent_bits(int hi) { return ((unsigned)hi >> 20) & 2047u; }
// the exponent field of an argument lies within 2^+-900
__device__ __forceinline__ bool common(unsigned e) { return e - 123u < 1801u; }

// Rounding by the remainder: the quotient's 53 bits are cut off a little below it (by
// BELOW of its last places, more than its error), so that the integer R is at most it and
// less than 1.5 short of it, and the remainder N - R D, which fits 64 bits and so needs
// only the products' lower halves, tells whether R or R + 1 is the nearest.
constexpr u64 BELOW = 8;

// 1 / x, x of either sign
__device__ __forceinline__ double recip64(double x) {
  const int h = __double2hiint(x);
  const unsigned e = exponent_bits(h);
  if (!common(e)) return div64_rare(1.0, x);
  const u64 m = significand(x);
  u64 r = (recip_q61(m) - BELOW) >> 8;                                      // 2^105 / m
  const i64 rem = (i64)(0 - r * m);
  r += 2 * rem > (i64)m ? 1 : 0;
  return __longlong_as_double((i64)(((u64)(2044 - e) << 52) + r) | ((i64)h & 0x80000000ll) << 32);
}

// a / b, of either sign
__device__ __forceinline__ double div64(double a, double b) {
  const int ha = __double2hiint(a), hb = __double2hiint(b);
  const unsigned ea = exponent_bits(ha), eb = exponent_bits(hb);
  if (!(common(ea) && common(eb) && ea - eb + 900u < 1801u)) return div64_rare(a, b);
  const u64 ma = significand(a), mb = significand(b);
  const u64 q = __umul64hi(ma << 11, recip_q61(mb));                        // in (1/2, 2), Q60
  const bool low = q < (1ull << 60);
  u64 r = (q - BELOW) >> (low ? 7 : 8);                                     // 2^53 ma / mb or half that
  const i64 rem = (i64)((ma << (low ? 53 : 52)) - r * mb);
  r += 2 * rem > (i64)mb ? 1 : 0;
  return __longlong_as_double((i64)(((u64)(1022 + ea - eb - (low ? 1u : 0u)) << 52) + r) |
                              ((i64)(ha ^ hb) & 0x80000000ll) << 32);
}

// the significand times 2^(exponent parity), Q62, in FP32, and half the exponent
struct RootArg {
  u64 m;
  float f;
  int half;
  bool ok;
};
__device__ __forceinline__ RootArg root_arg(double x) {
  RootArg a;
  const int h = __double2hiint(x);
  const int e = (h >> 20) - 1023;
  const u64 m = significand(x);
  a.ok = common((unsigned)(h >> 20));              // (a negative x: out of range)
  a.m = m << (10 + (e & 1));
  a.f = __uint_as_float((0x3f800000u + ((unsigned)(e & 1) << 23)) | ((unsigned)(m >> 29) & 0x7fffffu));
  a.half = e >> 1;
  return a;
}
// x^(-1/2)
__device__ __forceinline__ double rsqrt64(double x) {
  const RootArg a = root_arg(x);
  if (!a.ok) return rsqrt64_rare(x);
  const u64 r = (rsqrt_q61(a.m, a.f) + 128) >> 8;
  return __longlong_as_double((i64)(((u64)(1021 - a.half) << 52) + r));
}
// x^(1/2) = m m^(-1/2)
__device__ __forceinline__ double sqrt64(double x) {
  const RootArg a = root_arg(x);
  if (!a.ok) return __double_as_longlong(x) == 0ll ? 0.0 : sqrt64_rare(x);
  const u64 s = __umul64hi(a.m, rsqrt_q61(a.m, a.f));                       // in [1, 2], Q59
  u64 r = (s - BELOW) >> 7;
  const i64 rem = (i64)((a.m << 42) - r * r);                               // (r + 1/2)^2 = r^2 + r + 1/4
  r += rem > (i64)r ? 1 : 0;
  return __longlong_as_double((i64)(((u64)(1022 + a.half) << 52) + r));
}

// x 2^-k, exact
__device__ __forceinline__ double scale2(double x, int k) {
  const int h = __double2hiint(x), e = (int)exponent_bits(h);
  if (common((unsigned)e) && (unsigned)(e - k - 1) < 2046u)
    return __hiloint2double(h - k * 0x100000, __double2loint(x));
  return ldexp(x, -k);
}

// Conversions between FP64 and FP32, the narrowing one to nearest even, as the
// instructions do, which take the FP64 pipe
__device__ __forceinline__ float to_float(double x) {
  const unsigned h = (unsigned)__double2hiint(x), l = (unsigned)__double2loint(x);
  const int e = (int)exponent_bits((int)h) - 896;
  const unsigned r = ((unsigned)e << 23) + ((h & 0xfffffu) << 3 | l >> 29);
  const unsigned b = r + (((l & 0x1fffffffu) + 0x0fffffffu + (r & 1u)) >> 29) + (h & 0x80000000u);
  if ((unsigned)(e - 1) < 254u) return __uint_as_float(b);
  return (h << 1 | l) == 0u ? __uint_as_float(h) : (float)x;
}
__device__ __forceinline__ double to_double(float x) {
  const unsigned b = __float_as_uint(x);
  if ((b & 0x7f800000u) - 0x00800000u < 0x7f000000u)
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(b << 29));
  return (b << 1) == 0u ? __hiloint2double((int)b, 0) : (double)x;
}

// x^a for positive x by a table-driven logarithm and exponential (the method of Tang, ACM
// TOMS 15 (1989) 144 and 16 (1990) 378):
//   x = 2^e m, 1 <= m < 2, c from a table a little above 1/m, r = m c - 1 >= 0 (exact),
//   log2 x = e + log2(1/c) + r (polynomial),  y = a log2 x in Q58,
//   x^a = 2^n 2^(k/128) 2^g,  n + k/128 + g = y,  0 <= g < 1/128.
// Terms beyond the fourth (third) of the polynomials need 32 bits only.  |a| in
// [2^-6, 8); other a, and results beyond 2^+-1000, go to pow itself.
__device__ __forceinline__ double pow64(double x, double a) {
  const int hx = __double2hiint(x), ha = __double2hiint(a);
  const int e = (hx >> 20) - 1023, ea = (int)exponent_bits(ha) - 1023;
  const u64 m = significand(x);
  const unsigned k0 = (unsigned)(hx >> 13) & 127u;
  const ulonglong2 t0 = __ldg(reinterpret_cast<const ulonglong2*>(POW_LOG[k0]));
  const u64 r = m * (unsigned)t0.x << 1;                                    // Q64
  const unsigned r32 = (unsigned)(r >> 32);
  unsigned q32 = 0x2e2a8ecau;                                            // 1 / (j ln 2), j = 8 .. 1
  q32 = 0x34c2ec55u - __umulhi(q32, r32);
  q32 = 0x3d8e13b8u - __umulhi(q32, r32);
  q32 = 0x49ddb144u - __umulhi(q32, r32);
  u64 q = 0x171547652b82fe17ull - __umul64hi((u64)q32 << 30, r);
  q = 0x1ec709dc3a03fd75ull - __umul64hi(q, r);
  q = 0x2e2a8eca5705fc2full - __umul64hi(q, r);
  q = 0x5c551d94ae0bf85eull - __umul64hi(q, r);
  const u64 l = t0.y + __umul64hi(q, r);                                    // Q62
  // y = |a| (e + l): |a| = 2^ea ma
  const u64 ma = significand(a);
  const int sh = (2 - ea) & 15;
  const u64 al = __umul64hi(l, ma << 10) >> sh;                             // Q58
  const u64 as = ma << 8 >> sh;                                             // |a|, Q58 (exact)
  u64 lo = (u64)(i64)e * as;
  i64 hi = __mul64hi((i64)e, (i64)as);
  lo += al;
  hi += lo < al ? 1 : 0;
  if (ha < 0) {
    lo = 0 - lo;
    hi = ~hi + (lo == 0 ? 1 : 0);
  }
  const int kn = (int)((unsigned)(lo >> 51) | (unsigned)hi << 13);
  const u64 g = (lo << 13) >> 7;                                            // Q64
  const unsigned g32 = (unsigned)(g >> 32);
  unsigned p32 = 0x000a1849u;                                            // (ln 2)^j / j!, j = 6 .. 1
  p32 = 0x00576200u + __umulhi(p32, g32);
  p32 = 0x0276556eu + __umulhi(p32, g32);
  u64 p = 0x038d611ae09417f1ull + __umul64hi((u64)p32 << 30, g);
  p = 0x0f5fdeffc162c754ull + __umul64hi(p, g);
  p = 0x2c5c85fdf473de6bull + __umul64hi(p, g);
  p = __umul64hi(p, g);                                                     // 2^g - 1, Q62
  const u64 t1 = __ldg(&POW_EXP[kn & 127]);
  const u64 z = ((t1 >> 2) + __umul64hi(t1, p) + 128) >> 8;                 // from Q60, in [1, 2]
  const bool ok = common((unsigned)(hx >> 20)) && (unsigned)(ea + 6) < 9u &&
                  (unsigned)(kn + 128000) < 256000u;
  return ok ? __longlong_as_double((i64)(((u64)(i64)(1022 + (kn >> 7)) << 52) + z)) : pow64_rare(x, a);
}

}  // namespace amm
