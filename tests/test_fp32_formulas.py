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
