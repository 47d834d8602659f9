"""Reciprocal, exponentials and powers of the FP64 physics (csrc/dg_math64.cuh) on the device, against long double."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2306_01085_gb300", "csrc")
SOURCE = r"""
#include "dg_math64.cuh"
__global__ void k_math(int op, long long n, const double* x, const double* u, const double* v, double* y, double* z) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  if (op == 0) y[i] = dg::recip_fast(x[i]);
  else if (op == 1) y[i] = dg::exp_fast(x[i]);
  else if (op == 2) dg::exp_pm_fast(x[i], y[i], z[i]);
  else y[i] = dg::power_fast(x[i], u[i], v[i]);
}
extern "C" int run(int op, long long n, const double* x, const double* u, const double* v, double* y, double* z) {
  k_math<<<(unsigned)((n + 255) / 256), 256>>>(op, n, x, u, v, y, z);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def device(tmp_path_factory):
    import torch
    from paper_2306_01085_gb300 import build as B
    d = tmp_path_factory.mktemp("math64")
    (d / "m.cu").write_text(SOURCE)
    subprocess.run([B._nvcc(), *B.ARCH, "-O3", "-std=c++17", "--expt-relaxed-constexpr", "-shared", "-Xcompiler", "-fPIC",
                    "-I", CSRC, str(d / "m.cu"), "-o", str(d / "m.so")], check=True, capture_output=True)
    lib = ctypes.CDLL(str(d / "m.so"))

    def run(op, x, u=None, v=None):
        t = [torch.from_numpy(np.ascontiguousarray(a if a is not None else x)).cuda() for a in (x, u, v)]
        y, z = torch.zeros_like(t[0]), torch.zeros_like(t[0])
        p = [ctypes.c_void_p(a.data_ptr()) for a in (*t, y, z)]
        assert lib.run(op, ctypes.c_longlong(x.size), *p) == 0
        return y.cpu().numpy(), z.cpu().numpy()
    return run


def _ulps(y, t):
    """|y - t| in units of the last place of t (t: long double, normal FP64 range)."""
    _, e = np.frexp(np.abs(t))
    return np.abs(y.astype(np.longdouble) - t) / np.ldexp(np.longdouble(1), e - 53)


SPECIAL = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.2250738585072014e-308, 1.7976931348623157e308])


def test_reciprocal_is_nearly_correctly_rounded(device):
    """Newton-Raphson from a seed good to 2^-20: after two steps 2^-80 before the last rounding, so 0.5 units and
    2^-26; all exponents and both signs, and both sides of the limits 2^-991 and 2^993 beyond which (as for 0,
    subnormal, Inf, NaN) it is the division, bit for bit."""
    g = np.random.default_rng(1)
    e = np.repeat(np.arange(-1022, 1024), 100)
    x = np.ldexp(1.0 + g.random(e.size), e) * g.choice([-1.0, 1.0], e.size)
    edge = np.array([np.nextafter(b, d) for b in (2.0 ** -991, 2.0 ** 993) for d in (0.0, np.inf)] + [2.0 ** -991, 2.0 ** 993])
    x = np.concatenate([x, edge, -edge, 1.0 + 2.0 ** -52 * np.arange(2000), 2.0 - 2.0 ** -52 * np.arange(1, 2000)])
    y, _ = device(0, x)
    fast = (np.abs(x) >= 2.0 ** -991) & (np.abs(x) < 2.0 ** 993)
    assert fast.sum() > 190000
    with np.errstate(all="ignore"):
        assert float(_ulps(y[fast], np.longdouble(1) / x[fast].astype(np.longdouble)).max()) <= 0.5 + 2.0 ** -20
        assert np.array_equal(y[~fast], 1.0 / x[~fast])
        s, _ = device(0, SPECIAL)
        assert np.array_equal(s, 1.0 / SPECIAL, equal_nan=True) and np.array_equal(np.signbit(s[:4]), np.signbit(1.0 / SPECIAL[:4]))


def test_exponentials_on_both_sides_of_their_range(device):
    """0.65 units inside |x| < 64 (tests/test_exp_fixed.py), CUDA's exponential (1 unit) from there on and for Inf, NaN."""
    g = np.random.default_rng(2)
    x = np.concatenate([g.uniform(-63.999, 63.999, 60000), g.uniform(-1, 1, 20000) * 1e-5, g.uniform(-700, 700, 40000),
                        [np.nextafter(64.0, 0), 64.0, np.nextafter(64.0, 100), -64.0, -np.nextafter(64.0, 0), 0.0, -0.0]])
    y, _ = device(1, x)
    p, m = device(2, x)
    t = x.astype(np.longdouble)
    bound = np.where(np.abs(x) < 64.0, 0.65, 1.0)
    for got, want in ((y, np.exp(t)), (p, np.exp(t)), (m, np.exp(-t))):
        assert np.all(_ulps(got, want) <= bound)
    s, _ = device(1, SPECIAL)
    with np.errstate(all="ignore"):
        assert np.array_equal(s, np.exp(SPECIAL), equal_nan=True)


def test_powers_on_both_sides_of_their_range(device):
    """u^a e^(-a v / 2): 1.2 units inside the fixed-point range; outside it exp(a (log u - v / 2)) with a unit each for the
    logarithm and the exponential and half a unit for the two roundings of the exponent; 0 and Inf at u = 0 and Inf,
    NaN for negative u."""
    g = np.random.default_rng(3)
    n = 60000
    a = np.where(np.arange(n) % 2 == 0, 0.69, g.random(n))
    a[::7] *= 1.7                                          # beyond 1 in part: the general path
    u = np.exp2(g.uniform(-1, 1, n) * np.where(np.arange(n) % 3 == 0, 60, 39))
    v = g.uniform(-1, 1, n) * np.where(np.arange(n) % 5 == 0, 90.0, 60.0)
    y, _ = device(3, a, u, v)
    L = np.log(u.astype(np.longdouble)) - v.astype(np.longdouble) / 2
    want = np.exp(a.astype(np.longdouble) * L)
    inside = (u >= 2.0 ** -40) & (u < 2.0 ** 41) & (np.abs(v) < 64.0) & (a > 0.0) & (a < 1.0)
    assert 10000 < inside.sum() < n - 10000
    rel = np.abs(y.astype(np.longdouble) - want) / want
    general = 2.0 ** -53 * (2 + np.abs(a) * (2 * np.abs(np.log(u)) + 2 * np.abs(L)))
    assert float(_ulps(y[inside], want[inside]).max()) <= 1.2
    assert np.all(rel[~inside] <= general[~inside])
    s, _ = device(3, np.full(4, 0.5), np.array([0.0, np.inf, -1.0, np.nan]), np.ones(4))
    assert s[0] == 0.0 and s[1] == np.inf and np.isnan(s[2]) and np.isnan(s[3])
