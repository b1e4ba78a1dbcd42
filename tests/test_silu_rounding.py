"""The training kernel's SiLU and its derivative (csrc/mlp.cu), compiled for the
host with the reciprocal approximation moved by -1, 0 or +1 ulp: the quotients
z / q and 1 / q of the same FP32 q are the nearest floats (half an ulp, plus the
remainder's correction, whose own rounding is below 2^-20 ulp), the derivative
within the roundings of s (1 + z (1 - s)) from the nearest s."""
import re
import shutil
import subprocess
from pathlib import Path

import pytest

CSRC = Path(__file__).resolve().parent.parent / "paper_0901_4107_gb300" / "csrc"

MAIN = r"""
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#define __device__
#define __forceinline__ inline
static std::mt19937 rg(3);
static float ulps(float y, int k) { unsigned u; memcpy(&u, &y, 4); u += k; memcpy(&y, &u, 4); return y; }
static float approx_rcp(float x) { return ulps((float)(1.0 / (double)x), (int)(rg() %% 3) - 1); }
static float max_nan(float a, float b) { return a != a ? a : (a > b ? a : b); }
#define __expf exp_f
static float __expf(float x) { return (float)std::exp((double)x); }
static float __fmaf_rn(float a, float b, float c) { return std::fma(a, b, c); }
%s
static double err(float y, double r) { int e; std::frexp(r, &e); return std::fabs(((double)y - r) / std::ldexp(1.0, e - 24)); }
int main() {
  double eh = 0, ed = 0;
  for (long n = 0; n < 4000000; n++) {
    const double u = (double)rg() / 4294967296.0;
    float z = (float)(n %% 3 == 0 ? -87 + 160 * u : (n %% 3 == 1 ? 16 * u - 8 : 2 * u - 1));
    float h, d;
    silu_both(z, h, d);
    const float q = 1.0f + __expf(-z);
    if (z != 0) eh = std::fmax(eh, err(h, (double)z / q));
    const float s = (float)(1.0 / (double)q);
    const double t = 1.0 + (double)z * (1.0 - (double)s);
    // 1 - s: half an ulp of s or less; the sum's own rounding; the product's
    ed = std::fmax(ed, std::fabs(d - s * t) / (s * (std::fabs(z) + 2 * std::fabs(t)) * 0x1p-24 + 1e-44));
  }
  float h, d;
  int bad = 0;
  for (float z : {-87.5f, -100.0f, -1e4f, -3e38f}) {
    silu_both(z, h, d);
    bad += !(std::fabs(h) < 2e-36f && std::fabs(d) < 2e-36f);
  }
  for (float z : {87.5f, 200.0f, 1e30f}) {
    silu_both(z, h, d);
    bad += !(h == z && d == 1.0f);
  }
  silu_both(NAN, h, d);
  bad += h == h || d == d;
  std::printf("%%.9f %%.6f %%d\n", eh, ed, bad);
}
"""


def test_quotients_are_rounded_once(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    text = (CSRC / "mlp.cu").read_text()
    body = re.search(r"__device__ __forceinline__ void silu_both\(.*?\n}\n", text, re.S)[0]
    src = tmp_path / "silu.cpp"
    src.write_text(MAIN % body)
    exe = tmp_path / "silu"
    subprocess.run([gxx, "-O2", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    eh, ed, bad = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert float(eh) <= 0.5 + 2.0 ** -20 and float(ed) <= 1.0 and int(bad) == 0
    assert "__fdividef" not in text
