"""The integer FP64 <-> FP32 conversions that stand for the cvt instructions (csrc/dg_bits.cuh), compiled for the
host: to_f32_rn rounds to nearest even wherever to_f32_plain allows it, to_f64_exact is exact for every float."""
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_2306_01085_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include <cstring>
#include "dg_bits.cuh"
int main() {
  uint64_t b;
  while (scanf("%llx", (unsigned long long*)&b) == 1) {
    double d; memcpy(&d, &b, 8);
    float f = dg::to_f32_rn(d), g;
    uint32_t low = (uint32_t)b, fb; memcpy(&fb, &f, 4); memcpy(&g, &low, 4);
    double w = dg::to_f64_exact(g);
    uint64_t wb; memcpy(&wb, &w, 8);
    printf("%d %08x %016llx\n", (int)dg::to_f32_plain(d), fb, (unsigned long long)wb);
  }
  return 0;
}
"""


def test_conversions_match_ieee(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime.h")):
        pytest.skip("needs a host C++ compiler and the CUDA headers")
    (tmp_path / "x.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-O1", "-std=c++17", "-I", CSRC, "-I", inc, str(tmp_path / "x.cpp"), "-o", str(tmp_path / "x")],
                   check=True, capture_output=True)
    rng = np.random.default_rng(3)
    f = rng.integers(0, 2 ** 32, 4000, dtype=np.uint64)      # floats of every kind
    edge = np.array([0, 1, 0x7fffff, 0x800000, 0x7f7fffff, 0x7f800000, 0x7f800001, 0x7fc00000], dtype=np.uint64)
    f = np.concatenate([f, edge, edge | 0x80000000])
    with np.errstate(invalid="ignore"):
        base = f.astype(np.uint32).view(np.float32).astype(np.float64).view(np.uint64)
    # a float's double, its neighbours, the halfway points and their neighbours, in both low words
    d = np.concatenate([base + k for k in (0, 1, 2 ** 28 - 1, 2 ** 28, 2 ** 28 + 1)] +
                       [rng.integers(0, 2 ** 64, 4000, dtype=np.uint64)])
    d = np.concatenate([d, d >> np.uint64(32), f])           # low words that are floats as well
    out = subprocess.run([str(tmp_path / "x")], input="\n".join("%x" % int(x) for x in d), capture_output=True,
                         text=True, check=True).stdout.split()
    plain = np.array([int(x) for x in out[0::3]], dtype=bool)
    got32 = np.array([int(x, 16) for x in out[1::3]], dtype=np.uint32)
    got64 = np.array([int(x, 16) for x in out[2::3]], dtype=np.uint64)
    x = d.view(np.float64)
    with np.errstate(over="ignore", invalid="ignore"):
        want32 = x.astype(np.float32)
        size = np.abs(x)
        assert np.array_equal(plain, (x == 0) | ((size >= 2.0 ** -126) & (size < 2.0 ** 128)))
    assert plain.sum() > 10000 and np.array_equal(got32[plain], want32.view(np.uint32)[plain])
    low = d.astype(np.uint32).view(np.float32)
    with np.errstate(invalid="ignore"):
        want64 = low.astype(np.float64)
    nan = np.isnan(low)
    assert np.array_equal(got64[~nan], want64.view(np.uint64)[~nan]) and np.isnan(got64.view(np.float64)[nan]).all()
