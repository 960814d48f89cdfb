"""The mixed path's FP32 formulas against 64 bits, on the host: the device
headers compiled by the host compiler without contraction."""
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
// p: the pressure of recover_t; q: the FP64 balance of the same ke + me, rounded once
extern "C" void run_recover(long n, const float* u, const float* bl, const float* br, double gm1, float* p, float* q,
                            int* pairs) {
  for (long i = 0; i < n; ++i) {
    float w[8], eh, el, t;
    recover_t(u + 5 * i, bl + 3 * i, br + 3 * i, Gm1<float>(gm1), w);
    ke_me(u + 5 * i, bl + 3 * i, br + 3 * i, 1.0f / u[5 * i], eh, el);
    p[i] = w[4];
    q[i] = narrow_bits(gm1 * (widen_bits(u[5 * i + 4]) - (widen_bits(eh) + widen_bits(el))));
    pairs[i] = balance(u[5 * i + 4], eh, el, Gm1<float>(gm1), 0x1p-43f, t);
  }
}
template <int N> static void means(long n, const float* v, float* m, float* r) {
  for (long i = 0; i < n; ++i) {
    double d[N];
    for (int k = 0; k < N; ++k) d[k] = (double)v[8 * i + k];
    m[i] = mean<N>(v + 8 * i);
    r[i] = (float)mean<N>(d);
  }
}
extern "C" void run_mean(int N, long n, const float* v, float* m, float* r) {
  if (N == 2) means<2>(n, v, m, r);
  else if (N == 4) means<4>(n, v, m, r);
  else means<8>(n, v, m, r);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("fp32")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-fPIC", "-shared", "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_1110_1616_gb300", "csrc"), str(d / "t.cpp"), "-o", so], check=True)
    return C.CDLL(so)


def _p(a):
    return a.ctypes.data_as(C.c_void_p)


def _cells(n, rng, scale):
    """Cells of every kind: pressures from far below the energies to above them, exact cancellation, opposite faces,
    zero and non-finite values."""
    rho = np.exp(rng.uniform(-3, 3, n))
    v = rng.uniform(-1, 1, (n, 3)) * np.exp(rng.uniform(-6, 3, (n, 1)))
    bl = rng.uniform(-1, 1, (n, 3)) * np.exp(rng.uniform(-4, 2, (n, 1)))
    br = bl * (1 + 0.1 * rng.uniform(-1, 1, (n, 3)))
    br[::5] = -br[::5]
    u = np.column_stack([rho, rho[:, None] * v, np.zeros(n)]).astype(np.float32)
    bl, br = bl.astype(np.float32), br.astype(np.float32)
    ke = 0.5 * (u[:, 1:4].astype(float) ** 2).sum(1) / u[:, 0]
    me = 0.5 * ((0.5 * (bl.astype(float) + br)) ** 2).sum(1)
    p = np.exp(rng.uniform(-12, 3, n)) * np.where(np.arange(n) % 2, 1.0, ke + me)
    p[::97] = 0.0
    p[1::97] *= -1.0
    u[:, 4] = p * 1.5 + ke + me
    u[::7, 1:4] = 0.0
    f = np.float32(scale)
    u, bl, br = u * f, bl * np.sqrt(f), br * np.sqrt(f)
    for k, x in enumerate([np.nan, np.inf, -np.inf, 3e38, 0.0]):
        u[20 + 8 * k, 4] = x
        u[21 + 8 * k, 0] = x
        bl[22 + 8 * k, 1] = x
    return tuple(np.ascontiguousarray(x, np.float32) for x in (u, bl, br))


@pytest.mark.parametrize("scale", [1.0, 1e-12, 1e-25, 1e-33, 1e15, 1e33])
@pytest.mark.parametrize("gamma", [5.0 / 3.0, 1.4, 2.0])
def test_recovered_pressure_is_the_fp64_balance_bitwise(lib, scale, gamma):
    n = 400000
    u, bl, br = _cells(n, np.random.default_rng(int(10 * gamma)), scale)
    p, q, pairs = np.empty(n, np.float32), np.empty(n, np.float32), np.empty(n, np.int32)
    lib.run_recover(C.c_long(n), _p(u), _p(bl), _p(br), C.c_double(gamma - 1.0), _p(p), _p(q), _p(pairs))
    assert np.array_equal(p, q, equal_nan=True), np.flatnonzero(~((p == q) | (np.isnan(p) & np.isnan(q))))[:5]
    if 1e-20 < scale < 1e30:
        assert pairs.mean() > 0.9  # it is the pairs that are tested, not the FP64 line


@pytest.mark.parametrize("N", [2, 4, 8])
def test_mean_is_the_fp64_mean_rounded_once(lib, N):
    """Values within one binade (ties are common), spread over 2^16 and its edge, over all of FP32's range, with signs
    that cancel, zeros, infinities and NaN."""
    rng = np.random.default_rng(N)
    parts = [(1 + rng.integers(0, 2 ** 23, (200000, 8)) * 2.0 ** -23).astype(np.float32)]
    for spread in (3, 15, 16, 17, 30, 60, 250):
        x = np.exp2(rng.uniform(-spread / 2, spread / 2, (100000, 8))) * rng.choice([-1, 1], (100000, 8))
        x[::3, 1] = -x[::3, 0] * (1 + 2.0 ** -23 * rng.integers(-2, 3, len(x[::3])))
        parts.append(x.astype(np.float32))
    z = parts[1][:5000].copy()
    z[rng.random(z.shape) < 0.3] = 0.0
    s = (parts[1][:5000] * np.float32(2.0 ** -130)).astype(np.float32)
    e = parts[1][:5000].copy()
    e[rng.random(e.shape) < 0.1] = np.inf
    e[rng.random(e.shape) < 0.05] = np.nan
    e[rng.random(e.shape) < 0.1] = -np.inf
    big = (parts[0][:5000] * np.float32(1.5e38)).astype(np.float32)
    edge = np.float32(65536.0) * parts[0][:5000]
    edge[:, ::2] = parts[0][:5000, ::2]
    x = np.ascontiguousarray(np.concatenate(parts + [z, s, e, big, edge, np.zeros((8, 8), np.float32)]), np.float32)
    m, r = np.empty(len(x), np.float32), np.empty(len(x), np.float32)
    lib.run_mean(N, C.c_long(len(x)), _p(x), _p(m), _p(r))
    assert np.array_equal(m, r, equal_nan=True), np.flatnonzero(~((m == r) | (np.isnan(m) & np.isnan(r))))[:5]
