"""The FP64 kernels' restated formulas (HLLD flux, edge EMF, minmod, sign tests
on the bit patterns) against the formulas as written, bit for bit on the host:
the same device headers compiled by the host compiler without contraction."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cmath>
using std::fma; using std::fabs; using std::sqrt;
static inline unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) { return *p += v; }
#include "mhd_device.cuh"
using namespace amrdev;
template <class T> static T mm_written(T a, T b) {
  if (a > T(0) && b > T(0)) return (a <= b) ? a : b;
  if (a < T(0) && b < T(0)) return (a >= b) ? a : b;
  return T(0);
}
extern "C" void run_hlld(long n, const double* x, double gamma, double* f, double* g) {
  for (long i = 0; i < n; ++i) {
    hlld_flux<double>(x + 15 * i, x + 15 * i + 7, x[15 * i + 14], gamma, 1.0 / (gamma - 1.0), f + 7 * i);
    hlld_plain<double>(x + 15 * i, x + 15 * i + 7, x[15 * i + 14], gamma, 1.0 / (gamma - 1.0), g + 7 * i);
  }
}
extern "C" void run_emf(long n, const double* x, double* f, double* g) {
  for (long i = 0; i < n; ++i) {
    const double* y = x + 12 * i;
    f[i] = gs_emf<double>(y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[7], y[8], y[9], y[10], y[11]);
    g[i] = gs_emf_plain<double>(y[0], y[1], y[2], y[3], y[4], y[5], y[6], y[7], y[8], y[9], y[10], y[11]);
  }
}
extern "C" void run_pairs(long n, const double* a, const double* b, double* m, double* w, int* bad) {
  for (long i = 0; i < n; ++i) {
    const double x = a[i], y = b[i];
    m[i] = mm<double>(x, y);
    w[i] = mm_written<double>(x, y);
    const double py = fabs(y);
    bad[i] = (gt_zero(x) != (x > 0)) | (lt_zero(x) != (x < 0)) << 1 | (ge_zero(x) != (x >= 0)) << 2 |
             (le_zero(x) != (x <= 0)) << 3 | (gt_bits(x, y) != (x > y)) << 4 | (le_pos(py, x) != (py <= x)) << 5 |
             (abs_le(x, py) != (fabs(x) <= py)) << 6;
  }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp64")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_1110_1616_gb300", "csrc"), str(d / "t.cpp"), "-o", so], check=True)
    return C.CDLL(so)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _faces(n, rng):
    """Rotated face states of every HLLD region: smooth pairs, strong jumps,
    supersonic, weak and zero fields, equal sides, negative pressures, NaN."""
    x = np.empty((n, 15))
    for s in (0, 7):
        x[:, s] = np.exp(rng.uniform(-4, 4, n))
        x[:, s + 1:s + 4] = rng.normal(0, 1, (n, 3)) * np.exp(rng.uniform(-3, 3, (n, 1)))
        x[:, s + 4] = np.exp(rng.uniform(-4, 4, n))
        x[:, s + 5:s + 7] = rng.normal(0, 1, (n, 2)) * np.exp(rng.uniform(-4, 2, (n, 1)))
    x[:, 14] = rng.normal(0, 1, n) * np.exp(rng.uniform(-4, 2, n))
    k = n // 8
    x[:k, 7:14] = x[:k, :7] * (1 + 1e-3 * rng.normal(size=(k, 7)))  # smooth
    x[k:2 * k, 7:14] = x[k:2 * k, :7]                               # equal sides
    x[2 * k:3 * k, 14] = 0.0
    x[3 * k:4 * k, 14] *= 1e-9
    x[4 * k:4 * k + k // 2, [5, 6, 12, 13, 14]] = 0.0               # no field at all
    x[5 * k:5 * k + k // 2, 1:4] = 0.0                              # at rest
    x[5 * k:5 * k + k // 2, 8:11] = 0.0
    j = slice(6 * k, 6 * k + k // 4)
    x[j, 4] *= -1.0                                                 # negative predicted pressure
    x[6 * k + k // 4, 0] = np.nan
    x[6 * k + k // 4 + 1, 8] = np.nan
    return np.ascontiguousarray(x)


def test_hlld_flux_fp64_bitwise(lib):
    rng = np.random.default_rng(0)
    x = _faces(160000, rng)
    f, g = np.empty((len(x), 7)), np.empty((len(x), 7))
    lib.run_hlld(C.c_long(len(x)), _p(x), C.c_double(5.0 / 3.0), _p(f), _p(g))
    assert np.array_equal(f, g, equal_nan=True)
    assert np.isfinite(g).mean() > 0.95


def test_edge_emf_fp64_bitwise(lib):
    rng = np.random.default_rng(1)
    x = rng.normal(size=(100000, 12))
    x[::7, 8] = 0.0
    x[::11, 9:] = 0.0
    x[5::13, 10] = -0.0
    x[3, 8] = np.nan
    f, g = np.empty(len(x)), np.empty(len(x))
    lib.run_emf(C.c_long(len(x)), _p(x), _p(f), _p(g))
    assert np.array_equal(f, g, equal_nan=True)


def test_minmod_and_comparisons_bitwise(lib):
    sp = np.array([0.0, -0.0, 5e-324, -5e-324, 2.2e-308, 1.0, -1.0, 1.0 + 2 ** -52, 1.8e308, -1.8e308, np.inf, -np.inf,
                   np.nan, -np.nan, 1e-200, -1e-200])
    a, b = (v.ravel() for v in np.meshgrid(sp, sp))
    rng = np.random.default_rng(2)
    r = rng.integers(0, 2 ** 64, size=(2, 200000), dtype=np.uint64).view(np.float64)
    a = np.ascontiguousarray(np.concatenate([a, r[0], rng.normal(size=1000)]))
    b = np.ascontiguousarray(np.concatenate([b, r[1], np.zeros(1000)]))
    m, w, bad = np.empty_like(a), np.empty_like(a), np.empty(len(a), np.int32)
    lib.run_pairs(C.c_long(len(a)), _p(a), _p(b), _p(m), _p(w), _p(bad))
    assert not bad.any(), np.flatnonzero(bad)[:5]
    assert np.array_equal(m.view(np.uint64), w.view(np.uint64))
