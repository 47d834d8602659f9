"""The fixed-point exponentials and powers (csrc/dg_exp_fx.cuh), compiled for the host, against long double."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2306_01085_gb300", "csrc")

PROGRAM = r"""
#include <cmath>
#include <cstdio>
#include <random>
#include "dg_exp_fx.cuh"
static double ulps(double y, long double t) { int e; frexpl(t, &e); return (double)(fabsl(y - t) / ldexpl(1.0L, e - 53)); }
int main() {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  double we = 0, wp = 0, ww = 0;
  long done = 0;
  const double size[6] = {63.999, 8.0, 0.35, 2e-2, 1e-6, 1e-300};
  for (int i = 0; i < 600000; ++i) {
    double x = U(g) * size[i % 6];
    if (i < 40) x = (i - 20) * 0.0054152123481245726 * (i & 1 ? 1.0 : 1.0000000001);   // steps of the table
    double p, m;
    dg::fx_exp_pm(x, p, m);
    we = fmax(we, ulps(dg::fx_exp(x), expl((long double)x)));
    wp = fmax(wp, fmax(ulps(p, expl((long double)x)), ulps(m, expl(-(long double)x))));
    const double a = i & 1 ? 0.69 : fabs(U(g)), v = U(g) * (i % 3 ? 30.0 : 63.999), u = exp2(U(g) * (i % 3 ? 6 : 39.99));
    if (!dg::fx_power_range(a, u, v)) continue;
    ++done;
    ww = fmax(ww, ulps(dg::fx_power(a, u, v), expl((long double)a * (logl((long double)u) - (long double)v / 2))));
  }
  const double inf = INFINITY, out[] = {64.0, -64.0, 1e300, inf, -inf, NAN};
  int refused = 0;
  for (double x : out) refused += !dg::fx_exp_range(x) && !dg::fx_power_range(0.5, 1.0, x);
  for (double u : {0.0, -1.0, 4.4e12, 9e-13, inf, (double)NAN, 5e-324}) refused += !dg::fx_power_range(0.5, u, 1.0);
  for (double a : {0.0, 1.0, -0.5, (double)NAN}) refused += !dg::fx_power_range(a, 1.0, 1.0);
  printf("%f %f %f %ld %d %d\n", we, wp, ww, done, refused, dg::fx_exp(0.0) == 1.0 && dg::fx_exp(-5e-324) == 1.0);
  return 0;
}
"""


def test_errors_in_units_of_the_last_place(tmp_path):
    """Rounding 0.5, argument (2^-57) and series (2^-58) relative: 0.65; the logarithm's series (3 units of 2^-56),
    its constants and the product with a (one unit) on top: 1.2."""
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    if os.uname().machine != "x86_64":
        pytest.skip("the reference is the 80-bit long double")
    (tmp_path / "x.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", inc, str(tmp_path / "x.cpp"), "-o", str(tmp_path / "x")],
                   check=True, capture_output=True)
    out = subprocess.run([str(tmp_path / "x")], capture_output=True, text=True, check=True).stdout.split()
    assert float(out[0]) <= 0.65 and float(out[1]) <= 0.65 and float(out[2]) <= 1.2
    assert int(out[3]) > 500000 and int(out[4]) == 17 and int(out[5]) == 1
