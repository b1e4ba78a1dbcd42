"""csrc/fixed64.cuh compiled for the host with the hardware's FP32 approximations
anywhere within their documented errors (rcp.approx 1 ulp, rsqrt.approx a relative
2^-22.9, which is 2 ulp below 1): the reciprocal, quotient and square root are the
bits of IEEE 754's, at significands next to powers of two, next to ties, exact
squares, equal and neighbouring operands too; x^(-1/2) and x^a stay within 0.52 and
0.59 ulp of long double."""
import re
import shutil
import subprocess

import pytest

from tests.test_fixed64 import CSRC, SHIM

SEEDS = r"""
static inline float step(float y, int k) { unsigned u; memcpy(&u, &y, 4); return __uint_as_float(u + (unsigned)k); }
static int far = 0;   // the last seed's distance in ulps, for the report
static inline float seed_rcp(float x) {
  const float z = step((float)(1.0 / x), (int)(rg() % 3) - 1);
  return z > 1.0f ? 1.0f : z;
}
static inline float seed_rsqrt(float x) {
  const double t = 1.0 / std::sqrt((double)x);
  float z = step((float)t, (int)(rg() % 5) - 2);
  if (std::fabs(z - t) > t * 0x1.12p-23) z = (float)t;   // 2^-22.9
  if (std::fabs(z - t) > 0x1p-24) far++;
  return z > 1.0f ? 1.0f : z;
}
"""

MAIN = r"""
using namespace amm;
static double err(double y, long double r) {
  int e; std::frexp((double)r, &e);
  return (double)std::fabs((y - r) / (long double)std::ldexp(1.0, e - 53));
}
static double pick() {
  const int n = rg() % 6;
  double x = std::ldexp(1 + U(), (int)(rg() % 1600) - 800);
  if (n == 0) x = std::ldexp(1 + U() * 1e-9, (int)(rg() % 5) - 2);
  if (n == 1) x = std::nextafter(std::ldexp(1.0, (int)(rg() % 7) - 3), (rg() & 1) ? 0 : 1e9);
  if (n == 2) x = std::ldexp(1.0, (int)(rg() % 7) - 3);
  if (n == 3) { const double s = (double)(float)std::ldexp(1 + U(), (int)(rg() % 9) - 4); x = s * s; if (rg() & 1) x = std::nextafter(x, rg() & 1 ? 0 : 1e9); }
  if (n == 4) x = __longlong_as_double((__double_as_longlong(x) & ~0x1fffffffll) | (0x1fffffff - (long long)(rg() % 3)));   // the FP32 argument cut off most
  return x;
}
int main() {
  long bad[3] = {0, 0, 0};
  double m[2] = {0, 0};
  for (long n = 0; n < 3000000; n++) {
    const double x = pick();
    double a = std::ldexp(1 + U(), (int)(rg() % 80) - 40);
    const int c = rg() % 8;
    if (c == 0) a = x;
    if (c == 1) a = std::nextafter(x, rg() & 1 ? 0 : 1e300);
    if (c == 2) a = x * (1 + (double)(rg() % 1000) / 1024);
    // a quotient next to a tie: a = x (q + half an ulp), rounded
    if (c == 3) { const double q = 1 + U(); a = (double)((long double)x * ((long double)q + (long double)0x1p-53)); }
    bad[0] += recip64(x) != 1.0 / x || recip64(-x) != -1.0 / x;
    if (std::isnormal(a / x) && a / x > 1e-250 && a / x < 1e250) bad[1] += div64(a, x) != a / x || div64(-a, x) != -a / x;
    bad[2] += sqrt64(x) != std::sqrt(x);
    m[0] = std::fmax(m[0], err(rsqrt64(x), 1 / std::sqrt((long double)x)));
    const double g = 1.05 + 2 * U();
    const double es[4] = {(g - 1) / (2 * g), std::fmin(2 * g / (g - 1), 7.9), 1 / g, std::ldexp(1 + U(), (int)(rg() % 9) - 6)};
    const double p = es[rg() % 4] * ((rg() & 1) ? 1 : -1), b = std::exp((U() - 0.5) * 20);
    if (n % 4 == 0) m[1] = std::fmax(m[1], err(pow64(b, p), std::pow((long double)b, (long double)p)));
  }
  std::printf("%ld %ld %ld %.6f %.6f %d\n", bad[0], bad[1], bad[2], m[0], m[1], far);
}
"""


def test_rounded_as_ieee(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    text = (CSRC / "pow64_tables.cuh").read_text() + (CSRC / "fixed64.cuh").read_text()
    text = re.sub(r"(?m)^#(include|pragma).*$", "", text)
    text, n = re.subn(r"float y;\s*asm\(\"(rcp|rsqrt)\.approx[^\n]*\n\s*return y;", r"return seed_\1(x);", text)
    assert n == 2
    src = tmp_path / "fixed64.cpp"
    src.write_text(SHIM + SEEDS + text + MAIN)
    exe = tmp_path / "fixed64"
    subprocess.run([gxx, "-O2", "-w", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert [int(v) for v in out[:3]] == [0, 0, 0], out
    assert float(out[3]) <= 0.52 and float(out[4]) <= 0.59, out
    assert int(out[5]) > 1000   # seeds more than an ulp off were met
