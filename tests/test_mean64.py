"""The mean of eight children formed by integers (arith64.cuh) against the FP64
sums, bit for bit: both are one rounding to nearest even per sum."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = r"""
#include "arith64.cuh"
extern "C" void h_mean8(const double* v, long n, double* q) {
  for (long i = 0; i < n; ++i) {
    double x[8];
    for (int k = 0; k < 8; ++k) x[k] = v[8 * i + k];
    q[i] = mrb::mean8(x);
  }
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("mean64")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text("#include <cmath>\nnamespace mrb { static float seed_rcp(float x) { return 1.0f / x; }\n"
                   "static float seed_rsqrt(float x) { return 1.0f / std::sqrt(x); } }\n" + HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-Wno-unknown-pragmas",
                    "-Wno-unused-function", "-I", os.path.join(ROOT, "paper_2012_04385_gb300", "csrc"), str(src), "-o",
                    str(so)], check=True)
    return ctypes.CDLL(str(so))


@pytest.mark.parametrize("kind", ["one exponent", "low bits", "neighbouring exponents", "any", "equal", "zeros"])
def test_mean_of_eight_equals_the_sums(host, kind):
    rng = np.random.default_rng(3)
    n = 20_000
    frac = rng.integers(0, 1 << 52, (n, 8)).astype(np.uint64)
    # exponents over the whole range, each end included (0: subnormal, 2043 .. 2047: sums overflow, inf, NaN)
    e = rng.integers(0, 2048, (n, 1)).astype(np.uint64)
    e[: n // 2] = rng.choice(np.uint64([0, 1, 2, 1023, 2040, 2041, 2042, 2043, 2044, 2045, 2046, 2047]), (n // 2, 1))
    s = rng.integers(0, 2, (n, 1)).astype(np.uint64)
    if kind == "low bits":
        frac = (np.uint64((1 << 52) - 8) + rng.integers(0, 8, (n, 8)).astype(np.uint64)) * rng.integers(0, 2, (n, 1)).astype(
            np.uint64) + rng.integers(0, 4, (n, 8)).astype(np.uint64)
        frac &= np.uint64((1 << 52) - 1)
    if kind == "neighbouring exponents":
        e = np.clip(e.astype(np.int64) + rng.integers(0, 2, (n, 8)), 0, 2047).astype(np.uint64)
    if kind == "any":
        e, s = rng.integers(1000, 1050, (n, 8)).astype(np.uint64), rng.integers(0, 2, (n, 8)).astype(np.uint64)
    if kind == "equal":
        frac = np.repeat(frac[:, :1], 8, axis=1)
    if kind == "zeros":
        frac[:], e, s = 0, np.zeros((n, 1), np.uint64), rng.integers(0, 2, (n, 8)).astype(np.uint64)
    v = np.ascontiguousarray(((s << np.uint64(63)) | (e << np.uint64(52)) | frac).view(np.float64))
    got = np.empty(n)
    p = ctypes.POINTER(ctypes.c_double)
    host.h_mean8(v.ctypes.data_as(p), ctypes.c_long(n), got.ctypes.data_as(p))
    with np.errstate(all="ignore"):
        want = 0.125 * (((v[:, 0] + v[:, 1]) + (v[:, 2] + v[:, 3])) + ((v[:, 4] + v[:, 5]) + (v[:, 6] + v[:, 7])))
    nan = np.isnan(want)
    assert np.array_equal(np.isnan(got), nan)
    assert np.array_equal(got[~nan].view(np.uint64), want[~nan].view(np.uint64))
