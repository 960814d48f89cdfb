"""The launch shapes a level gets without amrmhd_autotune (the rule of
amrmhd_bind_arena): the results are those of 16x8 whole columns up to FP32
rounding, from one patch to many, even and ragged, with and without refined
levels, and the rule splits a level that does not fill the GPU."""
import numpy as np
import pytest

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


def problem(n, psize, refine):
    base = (n, n, n)
    patches = inputs.tile(0, (0, 0, 0), base, psize, 3)
    state = {0: inputs.blast_3d(n, n).state[0]}
    if refine:
        a, b = 2 * (n // 4), 2 * (3 * n // 4)
        patches += inputs.tile(1, (a, a, a), (b, b, b), psize, 3)
        state[1] = inputs.blast_3d(2 * n, 2 * n).state[0]
    return inputs.Problem("shape", 3, base, patches, 2 if refine else 1, state)


def run(pb, steps, **opts):
    import torch
    ctx = A.context_for(pb, precision=A.MIXED, stream=torch.cuda.Stream().cuda_stream)
    for k, v in opts.items():
        ctx.set_option(getattr(A, k), v)
    ctx.alloc_arena()
    torch.cuda.synchronize()
    ctx.load_state(pb.state)
    ctx.step(steps)
    return ctx


@pytest.mark.parametrize("n,psize,refine", [(16, 16, False), (24, 8, False), (44, 20, False), (24, 12, True),
                                            (40, 16, True), (32, 10, True)])
def test_default_shape_keeps_results(n, psize, refine):
    pb = problem(n, psize, refine)
    a, b = run(pb, 2), run(pb, 2, OPT_TILE=2, OPT_ZCHUNK=0)
    for l in range(pb.nlev):
        for kind in ((0, 1) if l else (0,)):
            t, z = a.tile_choice(l, kind)
            assert 1 <= t <= 4 and (z == -2 or 0 <= z <= 16)
            assert b.tile_choice(l, kind) == (2, 0)
    sa, sb = a.read_state(), b.read_state()
    for f in range(8):
        x, y = (np.concatenate([v.ravel() for v in s[f]]) for s in (sa, sb))
        # FP32 rounding of two steps against a field of unit size
        assert np.abs(x - y).max() <= 2e-5 * max(1.0, np.abs(y).max()), (f, np.abs(x - y).max())


def test_small_level_is_split():
    assert run(problem(16, 16, False), 1).tile_choice(0, 0)[1] in (2, 3, 4)
