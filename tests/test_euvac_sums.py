"""The EUVAC band sums (csrc/dg_euvac64.cuh), compiled for the host, against long double."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2306_01085_gb300", "csrc")

PROGRAM = r"""
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <random>
#include <stdint.h>
#include <string.h>
using std::max; using std::min; using std::fma; using std::exp;
static int __double2hiint(double d) { uint64_t b; memcpy(&b, &d, 8); return (int)(b >> 32); }
static int __double2loint(double d) { uint64_t b; memcpy(&b, &d, 8); return (int)b; }
static double __hiloint2double(int h, int l) { uint64_t b = ((uint64_t)(uint32_t)h << 32) | (uint32_t)l; double d; memcpy(&d, &b, 8); return d; }
static int __clzll(long long x) { return x ? __builtin_clzll(x) : 64; }
#include "dg_euvac.h"
#include "dg_euvac64.cuh"
using dg::EuvFx;
static double worst[4];                      // error over its bound: S0, S1 of one absorber, of four
template <int NS>
static void check(const EuvFx& X, const double w[4], double k) {
  long double r0 = 0, r1 = 0, d0 = 0, d1 = 0;
  for (int j = 0; j < X.n; ++j) {
    long double Phi = X.phi[0][j];
    if (NS == 4) { Phi = 0; for (int s = 0; s < 4; ++s) Phi += (long double)w[s] * X.phi[s][j]; }
    const long double a = X.B[j] * Phi * expl(-Phi * k);
    r0 += a; r1 += Phi * a; d0 += Phi * k * a; d1 += Phi * k * Phi * a;
  }
  double S0, S1;
  dg::euvac_sums<NS>(&X, w, k, S0, S1);
  auto put = [](double& to, double S, long double r, long double depth) {
    if (r < 1e-290L) to = std::max(to, fabsl(S - r) < 1e-300L ? 0.0 : 1e300);   // near the end of the FP64 range
    else to = std::max(to, (double)(fabsl(S - r) / r / (ldexpl(1.0L, -53) * (2 + depth / r))));
  };
  put(worst[NS == 1 ? 0 : 2], S0, r0, d0);
  put(worst[NS == 1 ? 1 : 3], S1, r1, d1);
}
int main() {
  double B[40], phi[4][40];
  for (int j = 0; j < dg::kEuvacRows; ++j) {
    const dg::EuvacRow& r = dg::kEuvac[j];
    B[j] = r.flux * 1e13 * 1.9e-25 / (0.5 * (r.lo + r.hi) * 1e-10);
    const double f[4] = {r.phi_o, r.phi_n2, r.phi_o2, r.phi_he};
    for (int s = 0; s < 4; ++s) phi[s][j] = f[s] * 1e-22;
  }
  EuvFx one, four;
  dg::build_euv(dg::kEuvacRows, B, phi, 1, &one);
  dg::build_euv(dg::kEuvacRows, B, phi, 4, &four);
  std::mt19937_64 g(3);
  std::uniform_real_distribution<double> U(0.0, 1.0);
  for (int i = 0; i < 200000; ++i) {
    const double k = i < 5 ? pow(10.0, 4 * i + 10) : pow(10.0, 12 + 13.5 * U(g));
    check<1>(one, nullptr, k);
    // compositions from mixed to nearly one constituent (fractions down to 1e-12, or none)
    double w[4], sum = 0;
    for (int s = 0; s < 4; ++s) sum += w[s] = i % 4 == 0 ? U(g) : i % 4 == 1 && s == i / 4 % 4 ? 0.0 : pow(10.0, -12 * U(g));
    for (int s = 0; s < 4; ++s) w[s] /= sum;
    check<4>(four, w, k);
  }
  // refused arguments take the FP64 loop, with its results
  int same = 0;
  const double odd[4][4] = {{1, 0, 0, -1e-3}, {1, NAN, 0, 0}, {0.7, 0.2, 0.1, 0}, {0.7, 0.2, 0.1, 0}};
  const double ks[4] = {1e20, 1e20, INFINITY, -1e20};
  for (int i = 0; i < 4; ++i) {
    double S0, S1, s0 = 0, s1 = 0;
    dg::euvac_sums<4>(&four, odd[i], ks[i], S0, S1);
    for (int j = 0; j < four.n; ++j) {
      double P = fma(odd[i][0], phi[0][j], fma(odd[i][1], phi[1][j], fma(odd[i][2], phi[2][j], odd[i][3] * phi[3][j])));
      const double a = (B[j] * P) * exp(-P * ks[i]);
      s0 += a; s1 = fma(P, a, s1);
    }
    same += (S0 == s0 || (std::isnan(S0) && std::isnan(s0))) && (S1 == s1 || (std::isnan(S1) && std::isnan(s1)));
  }
  printf("%g %g %g %g %d\n", worst[0], worst[1], worst[2], worst[3], same);
  return 0;
}
"""


def test_relative_error_at_any_depth_and_composition(tmp_path):
    """Both sums to a relative error of 2 + tau units of 2^-53, tau the mean optical depth of the bands that
    carry the sum: one unit for the conversion to FP64, one for the factors and the rounding of up to 40 terms at 2^-56, and the
    optical depth's own relative error below 2^-53 in the exponent."""
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
    assert all(float(x) <= 1.0 for x in out[:4]), out
    assert int(out[4]) == 4
