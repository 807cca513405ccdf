"""FP64 stage arithmetic on the host: the integer division and square root
(arith64.cuh) against IEEE, and the reordered face flux (flux64.cuh) against the
oracle's, bit for bit.  Both headers are plain C++ apart from two FP32 seeds,
for which the harness below takes values off by up to 2^-22 either way."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

import oracle

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HARNESS = r"""
#include <cmath>
#include <cstdint>
static double g_off = 0.0;
namespace mrb {
float seed_rcp(float x) { return (float)(1.0 / (double)x * (1.0 + g_off)); }
float seed_rsqrt(float x) { return (float)(1.0 / std::sqrt((double)x) * (1.0 + g_off)); }
}
#include "flux64.cuh"
using namespace mrb;
extern "C" {
void h_seed(double off) { g_off = off; }
void h_div(const double* a, const double* b, long n, double* q) { for (long i = 0; i < n; ++i) q[i] = div64(a[i], b[i]); }
void h_div6(const double* a, long n, double* q) { for (long i = 0; i < n; ++i) q[i] = div64_6(a[i]); }
void h_sqrt(const double* a, long n, double* q) { for (long i = 0; i < n; ++i) q[i] = sqrt64(a[i]); }
// U [n][6][5] lab frame -> F [n][5] lab frame; flat: the form for six equal cells
void h_flux(const double* U, long n, int d, double g, double B, int mode, int flux, int flat, double* F) {
  for (long i = 0; i < n; ++i) {
    double s[CQ_N * 6], f[5];
    for (int m = 0; m < 6; ++m) {
      const double* c = U + 30 * i + 5 * m;
      s[m] = c[0];
      for (int j = 0; j < 3; ++j) s[(1 + j) * 6 + m] = c[1 + (d + j) % 3];
      s[24 + m] = c[4];
      flux64_cell(d, g, B, s + m, 6);
    }
    const Row64 r{s, 6, 1};
    if (flat) face_flux64<true>(r, g, B, mode, flux, f);
    else face_flux64<false>(r, g, B, mode, flux, f);
    F[5 * i] = f[0];
    F[5 * i + 4] = f[4];
    for (int j = 0; j < 3; ++j) F[5 * i + 1 + (d + j) % 3] = f[1 + j];
  }
}
}
"""


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("flux64")
    src, so = d / "h.cpp", d / "h.so"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-Wno-unknown-pragmas", "-I",
                    os.path.join(ROOT, "paper_2012_04385_gb300", "csrc"), str(src), "-o", str(so)], check=True)
    L = ctypes.CDLL(str(so))
    vp, n, db, i = ctypes.c_void_p, ctypes.c_long, ctypes.c_double, ctypes.c_int
    L.h_seed.argtypes = [db]
    L.h_div.argtypes = [vp, vp, n, vp]
    L.h_div6.argtypes = L.h_sqrt.argtypes = [vp, n, vp]
    L.h_flux.argtypes = [vp, n, i, db, db, i, i, i, vp]
    return L


def p(a):
    return a.ctypes.data


def same_bits(got, ref):
    nan = np.isnan(ref)
    return np.array_equal(np.isnan(got), nan) and np.array_equal(got[~nan].view(np.uint64), ref[~nan].view(np.uint64))


def operands(seed, n=200_000):
    """Random mantissas over the whole exponent range, clustered mantissas
    (all ones, few bits), products (exact quotients) and their neighbours, and
    the special values."""
    r = np.random.Generator(np.random.Philox(key=seed))
    w = r.integers(0, 2**64, n, dtype=np.uint64)
    k = np.arange(n) % 4
    near = (w & np.uint64(0x800FFFFFFFFFFFFF)) | (r.integers(900, 1150, n, dtype=np.uint64) << np.uint64(52))
    w = np.where(k >= 1, near, w)
    low = (np.uint64(1) << r.integers(0, 53, n, dtype=np.uint64)) - np.uint64(1)
    w = np.where(k == 2, w & ~low, np.where(k == 3, w | low, w))
    x = w.view(np.float64).copy()
    special = [0.0, -0.0, 1.0, -1.0, np.inf, -np.inf, np.nan, 5e-324, 2.2250738585072014e-308, 1.7976931348623157e308]
    x[: len(special)] = special
    return x


@pytest.mark.parametrize("off", [0.0, 2.0**-22, -2.0**-22])
def test_division_and_root_are_correctly_rounded(host, off):
    host.h_seed(off)
    with np.errstate(all="ignore"):
        a, b = operands(1), operands(2)[::-1].copy()
        c = a * b
        for x, y in ((a, b), (c, b), (np.nextafter(c, np.inf), b), (np.nextafter(c, 0), a)):
            x, y = np.ascontiguousarray(x), np.ascontiguousarray(y)
            q = np.empty_like(x)
            host.h_div(p(x), p(y), len(x), p(q))
            assert same_bits(q, x / y)
            host.h_div6(p(x), len(x), p(q))
            assert same_bits(q, x / 6.0)
            for s in (x, x * x, np.nextafter(x * x, 0)):
                s = np.ascontiguousarray(s)
                host.h_sqrt(p(s), len(s), p(q))
                assert same_bits(q, np.sqrt(s))


def states(kind, seed, n=400):
    """Six-cell stencils [n][6][5]: rough, smooth, nearly flat, at rest (with
    both zeros), supersonic, with velocities down to the subnormal range, flat."""
    r = np.random.Generator(np.random.Philox(key=seed))
    base = np.stack([r.uniform(0.1, 2, n), *r.uniform(-1, 1, (3, n)), r.uniform(0.1, 2, n)], axis=1)
    amp = {"rough": 0.9, "smooth": 1e-2, "nearly flat": 1e-14}.get(kind, 0.3)
    if kind == "supersonic":
        base[:, 1:4] *= 5
    prim = base[:, None, :] * (1 + amp * r.uniform(-0.5, 0.5, (n, 6, 5)))
    if kind == "at rest":
        prim[..., 1:4] = np.where(r.random((n, 6, 3)) < 0.5, 0.0, -0.0)
    if kind == "tiny":
        prim[..., 1:4] *= np.ldexp(1.0, -r.integers(400, 1080, (n, 6, 3))) * (r.random((n, 6, 3)) < 0.7)
    if kind == "flat":
        prim[:] = base[:, None, :]
        prim[::3, :, 1:4] = 0.0
    rho, v, pr = prim[..., 0], prim[..., 1:4], prim[..., 4]
    U = np.empty_like(prim)
    U[..., 0] = rho
    U[..., 1:4] = rho[..., None] * v
    U[..., 4] = pr / 0.4 + 0.5 * rho * (v * v).sum(-1)
    return np.ascontiguousarray(U)


@pytest.mark.parametrize("kind", ["rough", "smooth", "nearly flat", "at rest", "supersonic", "tiny", "flat"])
@pytest.mark.parametrize("flux", [0, 1, 2])
@pytest.mark.parametrize("mode", [0, 2, 3, 4])
def test_face_flux_matches_the_oracle_bit_for_bit(host, mode, flux, kind):
    host.h_seed(0.0)
    U = states(kind, 10 * mode + flux)
    for d in range(3):
        ref = np.empty((len(U), 5))
        for i in range(len(U)):
            oracle.lib().orc_face_flux(p(U[i]), d, 1.4, 0.0, mode, flux, p(ref[i]))
        for flat in ([0, 1] if kind == "flat" else [0]):
            got = np.empty_like(ref)
            host.h_flux(p(U), len(U), d, 1.4, 0.0, mode, flux, flat, p(got))
            assert same_bits(got, ref)
