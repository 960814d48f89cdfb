"""The staged FP64 advance reading its halo from the neighbour patches'
interiors and stage arrays (AMRMHD_OPT_DIRECT_HALO with AMRMHD_OPT_ADVANCE 0)
against the same kernels on filled ghosts, bit for bit: a patch that is its own
neighbour, two and more patches per axis, unequal extents, the strict and the
contracted build, and the oracle."""
import numpy as np
import pytest

from helpers import compare_states, gpu_level_arrays, max_err, oracle_for
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


def run(pb, steps, direct, strict=True):
    import torch
    ctx = A.context_for(pb, precision=A.FP64, strict_fp64=strict, stream=torch.cuda.Stream().cuda_stream)
    ctx.set_option(A.OPT_DIRECT_HALO, direct)
    ctx.alloc_arena()
    torch.cuda.synchronize()
    ctx.load_state(pb.state)
    return ctx, ctx.step(steps)


def bricks(n, shape):
    """the blast on n^3 in patches of the given unequal extents"""
    pb = inputs.blast_3d(n, n)
    patches = [(0, (i, j, k), (i + shape[0], j + shape[1], k + shape[2]))
               for k in range(0, n, shape[2]) for j in range(0, n, shape[1]) for i in range(0, n, shape[0])]
    return inputs.Problem("bricks", 3, (n, n, n), patches, 1, pb.state)


@pytest.mark.parametrize("n,shape", [(8, (8, 8, 8)), (16, (8, 8, 8)), (24, (8, 12, 6)), (20, (10, 4, 20)),
                                     (32, (16, 16, 16)), (48, (16, 16, 16))])
@pytest.mark.parametrize("strict", [True, False])
def test_direct_equals_filled_bitwise(n, shape, strict):
    pb = bricks(n, shape)
    (a, da), (b, db) = run(pb, 3, 1, strict), run(pb, 3, 0, strict)
    assert np.array_equal(da, db)
    sa, sb = a.read_state(), b.read_state()
    for f in range(8):
        for p in range(len(pb.patches)):
            assert np.array_equal(sa[f][p], sb[f][p]), (f, p)


def test_direct_equals_oracle():
    pb = inputs.mhd_wave(3, 16, "fast", amp=1e-2, v0=(0.3, -0.2, 0.25), psize=8)
    ctx, dts = run(pb, 4, 1)
    o = oracle_for(pb)
    assert np.array_equal(dts, np.array([o.step() for _ in range(4)]))
    assert max_err(compare_states(gpu_level_arrays(ctx, pb), o.get_state(), pb)) <= 1e-12
