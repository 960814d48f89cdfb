"""The FP64 CFL reduction evaluates in FP64 only the cells whose FP32 estimate
can hold the maximum: its dt equals, bit for bit, the oracle's over all cells,
for states that stress the estimate (pressures far below the energy, dominant
fields, supersonic flow, scales far from 1 and outside FP32's range, one hot
cell among equals, equal cells), and a non-physical cell anywhere is still
reported."""
import numpy as np
import pytest

from helpers import oracle_for
from paper_1110_1616_gb300 import amrmhd as A
from paper_1110_1616_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1110_1616_gb300 import build
    build.build()


# spread of rho, v, p, B (standard deviations of their logarithm or value) and their scales
STATES = {"smooth": (0.01, 0.01, 0.01, 0.01, 1, 1, 1, 1), "wild": (1.0, 1.0, 1.0, 1.0, 1, 1, 1, 1),
          "cold": (0.5, 1.0, 2.0, 0.3, 1, 10, 1e-9, 1), "beta": (0.5, 0.3, 1.0, 1.0, 1, 1, 1e-6, 30),
          "supersonic": (0.5, 1.0, 0.5, 0.1, 1, 1e4, 1, 1), "no_field": (0.5, 0.5, 0.5, 0.0, 1, 1, 1, 0),
          "tiny": (0.5, 0.5, 0.5, 0.5, 1e-24, 1e6, 1e-12, 1e-6), "huge": (0.5, 0.5, 0.5, 0.5, 1e20, 1e3, 1e26, 1e13),
          "out_of_range": (0.5, 0.5, 0.5, 0.5, 1e-50, 1, 1e-50, 1e-25), "equal": (0, 0, 0, 0, 1, 1, 1, 1)}


def problem(name, dim, n, psize, hot=False):
    s = STATES[name]
    rng = np.random.default_rng(len(name) + 10 * dim + n)
    nz = n if dim == 3 else 1
    c = (nz, n, n)
    rho = s[4] * np.exp(s[0] * rng.normal(size=c))
    p = s[6] * np.exp(s[2] * rng.normal(size=c))
    v = [s[5] * (0.3 + s[1] * rng.normal(size=c)) for _ in range(3)]
    if hot:
        p[0, n // 2, n - 1] *= 3.0
    faces, cell = [], []
    for d in range(3):
        ax = 2 - d
        b = s[7] * (0.5 + s[3] * rng.normal(size=c))
        if d == 2 and dim == 2:
            faces.append(b)
            cell.append(b)
            continue
        f = np.concatenate([b, np.take(b, [0], axis=ax)], axis=ax)
        faces.append(f)
        m = f.shape[ax]
        cell.append(0.5 * (np.take(f, range(m - 1), axis=ax) + np.take(f, range(1, m), axis=ax)))
    e = p / (inputs.GAMMA - 1) + 0.5 * rho * sum(x * x for x in v) + 0.5 * sum(x * x for x in cell)
    base = (n, n, nz)
    return inputs.Problem(name, dim, base, inputs.tile(0, (0, 0, 0), base, psize, dim), 1,
                          {0: [rho, rho * v[0], rho * v[1], rho * v[2], e] + faces})


def context(pb, strict=True):
    import torch
    ctx = A.context_for(pb, precision=A.FP64, strict_fp64=strict, stream=torch.cuda.Stream().cuda_stream)
    ctx.alloc_arena()
    torch.cuda.synchronize()
    ctx.load_state(pb.state)
    return ctx


@pytest.mark.parametrize("dim,n,psize", [(2, 192, 192), (2, 256, 32), (2, 24, 6), (3, 36, 36), (3, 40, 10), (3, 20, 10)])
@pytest.mark.parametrize("name", list(STATES))
def test_dt_equals_the_oracle_bitwise(name, dim, n, psize):
    for hot in (False, True):
        pb = problem(name, dim, n, psize, hot)
        assert context(pb).cfl_dt() == oracle_for(pb).cfl_dt()


@pytest.mark.parametrize("field,value", [(0, -1.0), (0, np.nan), (4, 0.0), (4, np.nan), (1, np.inf)])
def test_a_bad_cell_is_reported(field, value):
    pb = problem("smooth", 3, 40, 10)
    pb.state[0][field][7, 3, 11] = value
    ctx = context(pb)
    with pytest.raises(A.AmrmhdError) as e:
        ctx.cfl_dt()
    assert e.value.status == A.ENONPHYS
