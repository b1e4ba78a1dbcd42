// x^a in FP64 for positive x: the power the wave curves need (fixed exponents,
// arguments of order one), by table-driven logarithm and exponential (the
// method of Tang, ACM TOMS 15 (1989) 144 and 16 (1990) 378):
//   x = 2^e m, 1 <= m < 2, c = 1/m to 9 bits from a table, r = m c - 1 (exact),
//   log2 x = (e + H) + (L + r (polynomial)),  H + L = log2(1/c), H on a grid,
//   a log2 x = hi + lo with hi = a (e + H) rounded and its remainder kept,
//   2^(hi + lo) = 2^n 2^(k/128) (1 + g (polynomial)), |g| <= 1/256.
// The remainders kept make the error that of the last rounding: at most 0.62
// ulp against 80-bit references over the tested range (CUDA's pow: 1 ulp by its
// documentation).  About 25 FP64 instructions; GB300 has one FP64 operation
// for 74 FP32 ones, and pow was most of the FP64 form's Riemann solve.
// Arguments outside (0, inf), subnormal ones and results beyond 2^+-1000 go
// to pow itself.
//
// Every operation is explicitly rounded, so the result is the same in every
// kernel that inlines it.
#pragma once

#include <cuda_runtime.h>

#include "pow64_tables.cuh"

namespace amm {

static __device__ __noinline__ double pow64_rare(double x, double a) { return pow(x, a); }

__device__ __forceinline__ double pow64(double x, double a) {
  const int hx = __double2hiint(x);
  // e + H, L, r
  const int k = (hx >> 13) & 127, e = (hx >> 20) - 1023;
  const double m = __hiloint2double((hx & 0xfffff) | 0x3ff00000, __double2loint(x));
  const double2 t0 = __ldg(reinterpret_cast<const double2*>(POW_LOG[k]));
  const double L = __ldg(&POW_LOG[k][2]);
  const double r = __fma_rn(m, t0.x, -1.0);
  double q = 0x1.a61762a7aded9p-3;                    // (-1)^(j+1) / (j ln 2), j = 7 .. 1
  q = __fma_rn(q, r, -0x1.ec709dc3a03fdp-3);
  q = __fma_rn(q, r, 0x1.2776c50ef9bfep-2);
  q = __fma_rn(q, r, -0x1.71547652b82fep-2);
  q = __fma_rn(q, r, 0x1.ec709dc3a03fdp-2);
  q = __fma_rn(q, r, -0x1.71547652b82fep-1);
  q = __fma_rn(q, r, 0x1.71547652b82fep+0);
  // e as a double without a conversion: 2^52 + 2^51 + e in the bits
  const double E = __dadd_rn(__hiloint2double(0x43380000, e), -0x1.8p52);
  const double h = __dadd_rn(E, t0.y);                // exact: H has 40 fractional bits
  const double l = __fma_rn(q, r, L);
  const double hi = __dmul_rn(a, h);
  const double lo = __fma_rn(a, l, __fma_rn(a, h, -hi));
  // hi + lo = n + k/128 + g
  const double s = __fma_rn(__dadd_rn(hi, lo), 128.0, 0x1.8p52);
  const int kn = __double2loint(s);
  const double g = __dadd_rn(__fma_rn(__dadd_rn(s, -0x1.8p52), -0x1p-7, hi), lo);
  const double2 t1 = __ldg(reinterpret_cast<const double2*>(POW_EXP[kn & 127]));
  double p = 0x1.430912f86c787p-13;                   // (ln 2)^j / j!, j = 6 .. 1
  p = __fma_rn(p, g, 0x1.5d87fe78a6731p-10);
  p = __fma_rn(p, g, 0x1.3b2ab6fba4e77p-7);
  p = __fma_rn(p, g, 0x1.c6b08d704a0c0p-5);
  p = __fma_rn(p, g, 0x1.ebfbdff82c58fp-3);
  p = __fma_rn(p, g, 0x1.62e42fefa39efp-1);
  p = __dmul_rn(p, g);
  const double y = __dadd_rn(t1.x, __fma_rn(t1.x, p, t1.y));
  const double z = __hiloint2double(__double2hiint(y) + ((kn >> 7) << 20), __double2loint(y));
  // (a comparison in integers: hi's exponent below 2^10, x normal and positive)
  const bool rare = (unsigned)(hx - 0x00100000) >= 0x7fe00000u ||
                    (unsigned)(__double2hiint(hi) & 0x7fffffff) >= 0x408f0000u;
  return rare ? pow64_rare(x, a) : z;
}

}  // namespace amm
