"""The FP64 wave curves f_K(p) of csrc/riemann.cuh, compiled for the host with the
fixed-point operations of csrc/fixed64.cuh, against long double: no further off, in
the mean square over shocks and rarefactions of any strength, than the formulas with
their plain quotients, root and power in FP64 (sqrt(A / (p + B)), (p / p_K)^z), and
within the sum of their own roundings, relative to f's terms: shock d, h, its
constant and p + B, their product (halved by the root), the root 0.52, the product;
rarefaction the quotient times z, the power 0.59, the difference, two products."""
import re
import shutil
import subprocess

import pytest

from tests.test_fixed64 import CSRC, SHIM

MAIN = r"""
namespace amm {
static double rn_mul(double a, double b) { return a * b; }
static double rn_add(double a, double b) { return a + b; }
static double rn_fma(double a, double b, double c) { return std::fma(a, b, c); }
static bool positive(double x) { return x > 0; }
template <typename T> struct GasC {
  T gm1_gp1, two_gm1, inv_g, z, half_gp1, two_gp1, sqrt_two_gp1;
  explicit GasC(double g) : gm1_gp1((g - 1) / (g + 1)), two_gm1(2 / (g - 1)), inv_g(1 / g), z((g - 1) / (2 * g)), half_gp1(0.5 * (g + 1)),
                            two_gp1(2 / (g + 1)), sqrt_two_gp1(std::sqrt(2 / (g + 1))) {}
};
%s
}  // namespace amm
using namespace amm;
int main() {
  double sn[2] = {0, 0}, sp[2] = {0, 0}, mx[2] = {0, 0};
  for (long n = 0; n < 800000; n++) {
    const double g = n %% 2 ? 5.0 / 3.0 : 1.4, rho = std::exp(6 * U() - 3), pK = std::exp(6 * U() - 3);
    const double ratio = n %% 3 == 0 ? std::exp(8 * U() - 4) : (n %% 3 == 1 ? 1 + 4 * U() : 0.3 + 0.7 * U());
    const double p = pK * ratio, c = std::sqrt(g * pK / rho);
    const GasC<double> G(g);
    double f, df;
    wave_curve(p, recip64(p), wave_side(rho, pK, c, G), G, f, df);
    const long double gl = g, pl = p, kl = pK, rl = rho;
    long double ex, scale;
    double plain;
    const int k = p > pK ? 0 : 1;
    if (k == 0) {
      ex = (pl - kl) * std::sqrt(2 / (gl + 1) / rl / (pl + (gl - 1) / (gl + 1) * kl));
      scale = ex;
      plain = (p - pK) * std::sqrt(G.two_gp1 / rho / (p + G.gm1_gp1 * pK));
    } else {
      const long double pr = std::pow(pl / kl, (gl - 1) / (2 * gl));
      ex = 2 / (gl - 1) * (long double)c * (pr - 1);
      scale = 2 / (gl - 1) * (long double)c;
      plain = G.two_gm1 * c * (std::pow(p / pK, G.z) - 1.0);
    }
    const double u = 0x1p-53L * scale, en = (double)((f - ex) / u), ep = (double)((plain - ex) / u);
    sn[k] += en * en;
    sp[k] += ep * ep;
    mx[k] = std::fmax(mx[k], std::fabs(en));
  }
  std::printf("%%.5f %%.5f %%.5f %%.5f\n", std::sqrt(sn[0] / sp[0]), std::sqrt(sn[1] / sp[1]), mx[0], mx[1]);
}
"""


def test_no_less_exact_than_the_formulas(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    strip = lambda t: re.sub(r"(?m)^#(include|pragma).*$", "", t)  # noqa: E731
    fixed = strip((CSRC / "pow64_tables.cuh").read_text() + (CSRC / "fixed64.cuh").read_text())
    fixed = re.sub(r"float y;\s*asm\(\"(rcp|rsqrt)\.approx[^\n]*\n\s*return y;",
                   lambda k: "return seed(1.0 / x);" if k[1] == "rcp" else "return seed(1.0 / std::sqrt((double)x));", fixed)
    text = (CSRC / "riemann.cuh").read_text()
    curve = text[text.index("struct WaveSide {"):text.index("// Linearised (primitive-variable) star pressure")]
    src = tmp_path / "wave.cpp"
    src.write_text(SHIM + fixed + MAIN % curve)
    exe = tmp_path / "wave"
    subprocess.run([gxx, "-O2", "-w", "-std=c++17", "-ffp-contract=off", "-o", str(exe), str(src)], check=True)
    shock, rare, ms, mr = [float(v) for v in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    # (a ratio of two sample deviations of 4e5 values: 0.5 %)
    assert shock <= 1.005 and rare <= 1.005, (shock, rare)
    # in half ulps' relative size 2^-53: d 1, [constant 1, h 1, B's product and sum 1, product 1] / 2, root 1.04, product 1
    assert ms <= 1 + 2 + 1.04 + 1 and mr <= 1 + 1.18 + 1 + 1 + 1, (ms, mr)


def test_the_sampled_density_is_one_power():
    text = (CSRC / "riemann.cuh").read_text()
    assert text.count("rhoF = rhoK * xpow(r, G.inv_g); uF = us; pF = ps;") == 1
