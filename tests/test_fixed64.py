"""The fixed-point FP64 reciprocal, quotient, square roots and power of
csrc/fixed64.cuh, and its conversions, compiled for the host with the two FP32 approximations
replaced by correctly rounded ones moved by -1, 0 or +1 ulp (their documented
error), against long double.

The bounds are half an ulp for the one rounding plus the truncations: the
reciprocal of a significand drops four terms of 2^-61 on a value above 1/2 (ulp
2^-53): 0.016; the quotient multiplies that by up to 2 and drops 2^-60: 0.03;
the root multiplies 2^-59 by m < 4 (ulp 2^-52): 0.04; the power's exponent y is
off by 8 x 2^-60 + 2^-58 (relative ulp 2^-53 at worst): 0.06 after ln 2, and its
exponential by 4 x 2^-60: 0.03."""
import re
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_0901_4107_gb300" / "csrc"
BOUND = {"recip": 0.516, "div": 0.53, "rsqrt": 0.52, "sqrt": 0.54, "pow": 0.59}

SHIM = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
#define __noinline__
struct ulonglong2 { unsigned long long x, y; };
static std::mt19937_64 rg(7);
static double U() { return (double)(rg() >> 11) * 0x1p-53; }
static inline float __uint_as_float(unsigned u) { float f; memcpy(&f, &u, 4); return f; }
static inline float seed(double v) {
  const float y = (float)v; unsigned u; memcpy(&u, &y, 4);
  const float z = __uint_as_float(u + (unsigned)((int)(rg() % 3) - 1));
  return z > 1.0f ? 1.0f : z;
}
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) { return (unsigned long long)(((unsigned __int128)a * b) >> 64); }
static inline long long __mul64hi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
static inline unsigned __umulhi(unsigned a, unsigned b) { return (unsigned)(((unsigned long long)a * b) >> 32); }
static inline long long __double_as_longlong(double d) { long long l; memcpy(&l, &d, 8); return l; }
static inline double __longlong_as_double(long long l) { double d; memcpy(&d, &l, 8); return d; }
static inline int __double2hiint(double d) { return (int)(__double_as_longlong(d) >> 32); }
static inline ulonglong2 __ldg(const ulonglong2* p) { return *p; }
static inline unsigned long long __ldg(const unsigned long long* p) { return *p; }
static inline unsigned __float_as_uint(float f) { unsigned u; memcpy(&u, &f, 4); return u; }
static inline int __double2loint(double d) { return (int)__double_as_longlong(d); }
static inline double __hiloint2double(int h, int l) { return __longlong_as_double((long long)h << 32 | (unsigned)l); }
static double rsqrt(double x) { return 1 / std::sqrt(x); }
"""

MAIN = r"""
using namespace amm;
static double err(double y, long double r) {
  int e; std::frexp((double)r, &e);
  return (double)std::fabs((y - r) / (long double)std::ldexp(1.0, e - 53));
}
int main() {
  double m[5] = {0, 0, 0, 0, 0};
  for (long n = 0; n < 1000000; n++) {
    double x = std::ldexp(1 + U(), (int)(rg() % 1600) - 800), a = std::ldexp(1 + U(), (int)(rg() % 80) - 40);
    if (n % 4 == 0) x = std::ldexp(1 + U() * 1e-9, (int)(rg() % 5) - 2);
    if (n % 4 == 1) x = std::nextafter(std::ldexp(1.0, (int)(rg() % 7) - 3), (rg() & 1) ? 0 : 1e9);
    if (n % 16 == 2) x = std::ldexp(1.0, (int)(rg() % 7) - 3);
    m[0] = std::fmax(m[0], err(recip64(x), 1.0L / x));
    m[0] = std::fmax(m[0], err(recip64(-x), -1.0L / x));
    m[1] = std::fmax(m[1], err(div64(-a, x), -(long double)a / x));
    m[2] = std::fmax(m[2], err(rsqrt64(x), 1 / std::sqrt((long double)x)));
    m[3] = std::fmax(m[3], err(sqrt64(x), std::sqrt((long double)x)));
    const double g = 1.05 + 2 * U();
    const double es[4] = {(g - 1) / (2 * g), std::fmin(2 * g / (g - 1), 7.9), 1 / g, std::ldexp(1 + U(), (int)(rg() % 9) - 6)};
    const double p = es[rg() % 4] * ((rg() & 1) ? 1 : -1);
    const double b = rg() % 3 ? std::exp((U() - 0.5) * 20) : (rg() & 1 ? 1 + (U() - 0.5) * 1e-6 : std::ldexp(1 + U(), (int)(rg() % 100) - 50));
    m[4] = std::fmax(m[4], err(pow64(b, p), std::pow((long double)b, (long double)p)));
  }
  std::printf("recip %.6f\ndiv %.6f\nrsqrt %.6f\nsqrt %.6f\npow %.6f\n", m[0], m[1], m[2], m[3], m[4]);
  // conversions and scaling: the same bits as the instructions', over all exponents, ties and neighbours of ties
  long bad = 0;
  for (long n = 0; n < 4000000; n++) {
    unsigned long long b = rg();
    if (n % 2) b = (b & 0x800fffffffffffffull) | (unsigned long long)(895 + rg() % 257) << 52;
    if (n % 8 == 3) b = (b & ~0x1fffffffull) | (0x10000000ull + rg() % 3 - 1);
    const double x = __longlong_as_double((long long)b);
    const float f = to_float(x), f0 = (float)x, h = __uint_as_float((unsigned)rg());
    const double d = to_double(h), d0 = (double)h;
    bad += !(f == f0 || (f != f && f0 != f0)) + !(d == d0 || (d != d && d0 != d0));
    const int k = (int)(rg() % 400) - 200;
    const double s = std::ldexp(1 + U(), (int)(rg() % 1200) - 600);
    bad += scale2(s, k) != std::ldexp(s, -k);
  }
  bad += std::signbit(to_float(-0.0)) == 0 || std::signbit(to_double(-0.0f)) == 0;
  std::printf("convert %ld\n", bad);
  // arguments outside the fixed-point ranges take the library's results
  const bool ok = recip64(0.0) == INFINITY && recip64(-INFINITY) == 0 && div64(0.0, 2.0) == 0 && std::isnan(div64(NAN, 1.0)) &&
                  sqrt64(0.0) == 0 && std::isnan(sqrt64(-1.0)) && rsqrt64(INFINITY) == 0 && pow64(0.0, 0.2) == 0 &&
                  std::isnan(pow64(NAN, 0.2)) && recip64(1e-310) == 1 / 1e-310 && sqrt64(1e-310) == std::sqrt(1e-310) &&
                  pow64(2.0, 9.0) == 512 && pow64(1e300, 7.9) == INFINITY && pow64(1.0, 7.0) == 1;
  std::printf("special %d\n", ok ? 0 : 1);
}
"""


def test_fixed_point_functions(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    text = (CSRC / "pow64_tables.cuh").read_text() + (CSRC / "fixed64.cuh").read_text()
    text = re.sub(r"(?m)^#(include|pragma).*$", "", text)
    text, n = re.subn(r"float y;\s*asm\(\"(rcp|rsqrt)\.approx[^\n]*\n\s*return y;",
                      lambda k: "return seed(1.0 / x);" if k[1] == "rcp" else "return seed(1.0 / std::sqrt((double)x));", text)
    assert n == 2
    src = tmp_path / "fixed64.cpp"
    src.write_text(SHIM + text + MAIN)
    exe = tmp_path / "fixed64"
    subprocess.run([gxx, "-O2", "-w", "-std=c++17", "-o", str(exe), str(src)], check=True)
    out = dict(line.split() for line in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.splitlines())
    assert float(out.pop("special")) == 0 and float(out.pop("convert")) == 0
    for name, bound in BOUND.items():
        assert float(out[name]) <= bound, (name, out)
