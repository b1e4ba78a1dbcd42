"""csrc/fixed64.cuh on the device, with the hardware's own approximations: the
reciprocal, quotient, square root and the conversions give the bits of CUDA's
operators, the reciprocal square root and the power stay within 0.52 and 0.59 ulp
of long double; arguments outside the fixed-point ranges give CUDA's results."""
import ctypes
import subprocess

import numpy as np
import pytest

from tests.test_fixed64 import CSRC

pytestmark = pytest.mark.gpu

SRC = r"""
#include "fixed64.cuh"
using namespace amm;
__global__ void k_all(int n, const double* x, const double* a, const double* p, double* o) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  o[i] = recip64(x[i]);
  o[n + i] = div64(a[i], x[i]);
  o[2 * n + i] = sqrt64(x[i]);
  o[3 * n + i] = rsqrt64(x[i]);
  o[4 * n + i] = pow64(x[i], p[i]);
  o[5 * n + i] = to_float(x[i]);
  o[6 * n + i] = to_double((float)a[i]);
  o[7 * n + i] = 1.0 / x[i];
  o[8 * n + i] = a[i] / x[i];
  o[9 * n + i] = sqrt(x[i]);
  o[10 * n + i] = rsqrt(x[i]);
  o[11 * n + i] = pow(x[i], p[i]);
  o[12 * n + i] = (float)x[i];
  o[13 * n + i] = (double)(float)a[i];
}
extern "C" int run(int n, const double* x, const double* a, const double* p, double* o) {
  k_all<<<(n + 255) / 256, 256>>>(n, x, a, p, o);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0901_4107_gb300 import _build
    d = tmp_path_factory.mktemp("fixed64")
    (d / "f.cu").write_text(SRC)
    so = d / "libf.so"
    subprocess.run([_build.nvcc(), "-shared", str(d / "f.cu"), "-o", str(so)] + _build.ARCH + _build.FLAGS, check=True)
    lib = ctypes.CDLL(str(so))

    def call(x, a, p):
        t = [torch.from_numpy(np.ascontiguousarray(v)).cuda() for v in (x, a, p)]
        o = torch.empty(14, len(x), dtype=torch.float64, device="cuda")
        torch.cuda.synchronize()
        assert lib.run(len(x), *[ctypes.c_void_p(v.data_ptr()) for v in t], ctypes.c_void_p(o.data_ptr())) == 0
        return o.cpu().numpy()
    return call


def ulps(y, r):
    return np.abs((y - r) / np.ldexp(np.longdouble(1), np.frexp(r.astype(np.float64))[1] - 53)).astype(np.float64)


def test_common_arguments(run):
    rng = np.random.default_rng(2)
    n = 1 << 20
    x = np.ldexp(1 + rng.random(n), rng.integers(-800, 800, n))
    x[::4] = np.ldexp(1 + rng.random(n // 4) * 1e-9, rng.integers(-2, 3, n // 4))
    x[1::8] = np.nextafter(np.ldexp(1.0, rng.integers(-3, 4, n // 8)), rng.choice([0.0, 1e9], n // 8))
    s = rng.random(n // 8).astype(np.float32).astype(np.float64) + 0.5
    x[3::8] = s * s
    a = np.ldexp(1 + rng.random(n), rng.integers(-40, 40, n)) * rng.choice([1.0, -1.0], n)
    a[5::8] = x[5::8]
    a[6::8] = np.nextafter(x[6::8], np.inf)
    g = 1.05 + 2 * rng.random(n)
    e = np.where(rng.random(n) < 0.5, (g - 1) / (2 * g), np.minimum(2 * g / (g - 1), 7.9)) * rng.choice([1.0, -1.0], n)
    xp = np.exp((rng.random(n) - 0.5) * 20)
    o = run(x, a, e)
    for k in (0, 1, 2):
        assert np.array_equal(o[k], o[7 + k])
    ok = np.abs(a) < 1e30
    assert np.array_equal(o[5], o[12]) and np.array_equal(o[6][ok], o[13][ok])
    assert ulps(o[3], 1 / np.sqrt(x.astype(np.longdouble))).max() <= 0.52
    o = run(xp, a, e)
    assert ulps(o[4], xp.astype(np.longdouble) ** e.astype(np.longdouble)).max() <= 0.59


def test_other_arguments(run):
    v = np.array([0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 1e-310, 1e308, 2.0 ** -1022, 2.0 ** 1023, -3.5, 1e-290])
    x, a = (m.ravel() for m in np.meshgrid(v, v))
    p = np.resize([0.2, -0.2, 2.5, 5.0, 9.0, 1e-3], len(x))
    o = run(x, a, p)
    for k in range(7):
        assert np.array_equal(o[k], o[7 + k], equal_nan=True), k
        z = o[7 + k] == 0
        assert np.array_equal(np.signbit(o[k][z]), np.signbit(o[7 + k][z])), k
