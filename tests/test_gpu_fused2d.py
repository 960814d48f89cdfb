"""The fused 2D advance of the mixed path (AMRMHD_OPT_ADVANCE 0) against the
staged kernels (2): tiles at the edges of their range (one cell more and less
than a tile, ragged and unequal patches, one patch and many), with and without
refined levels and physical boundaries, and the conserved totals, which the
registers (fed from the fluxes the fused kernel leaves) keep to FP32 rounding."""
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


def smooth(n, psize, refine):
    base = (n, n, 1)
    patches = inputs.tile(0, (0, 0, 0), base, psize, 2)
    if refine:
        a, b = 2 * (n // 4), 2 * (3 * n // 4)
        patches += inputs.tile(1, (a, a, 0), (b, b, 1), psize, 2)
    nlev = 2 if refine else 1
    return inputs.Problem("smooth2d", 2, base, patches, nlev, inputs.random_smooth_2d(n, nlev, seed=n))


PROBLEMS = {"%d_%d%s" % c: (lambda c=c: smooth(c[0], c[1], c[2] == "r"))
            for c in [(16, 16, ""), (18, 18, ""), (19, 19, ""), (36, 36, ""), (64, 11, ""), (8, 8, ""), (256, 32, ""),
                      (16, 8, "r"), (32, 32, "r"), (28, 14, "r"), (24, 6, "r"), (48, 20, "r"), (128, 32, "r")]}
PROBLEMS["orszag_tang"] = lambda: inputs.orszag_tang(64, 16, True)
PROBLEMS["bounded"] = lambda: inputs.smooth_bounded_2d(32, refine=True, seed=2)
PROBLEMS["clumps"] = lambda: inputs.clumps_2d()


def run(pb, steps, advance, graph=1):
    import torch
    ctx = A.context_for(pb, precision=A.MIXED, stream=torch.cuda.Stream().cuda_stream)
    ctx.set_option(A.OPT_ADVANCE, advance)
    ctx.set_option(A.OPT_GRAPH, graph)
    ctx.alloc_arena()
    torch.cuda.synchronize()
    ctx.load_state(pb.state)
    return ctx, ctx.step(steps)


@pytest.mark.parametrize("name", list(PROBLEMS))
def test_fused_equals_staged_up_to_rounding(name):
    pb = PROBLEMS[name]()
    (a, da), (b, db) = run(pb, 2, 0), run(pb, 2, 2)
    assert np.abs(da - db).max() <= 2e-6 * np.abs(db).max()
    sa, sb = a.read_state(), b.read_state()
    for f in range(8):
        x, y = (np.concatenate([v.ravel() for v in s[f]]) for s in (sa, sb))
        # FP32 rounding of two steps: a few hundred ulps of the field's size
        assert np.abs(x - y).max() <= 2e-5 * max(1.0, np.abs(y).max()), (f, np.abs(x - y).max())


def test_plain_launches_and_graph_are_the_same_bits():
    pb = PROBLEMS["128_32r"]()
    (a, da), (b, db) = run(pb, 3, 0, 1), run(pb, 3, 0, 0)
    assert np.array_equal(da, db)
    sa, sb = a.read_state(), b.read_state()
    for f in range(8):
        for p in range(len(pb.patches)):
            assert np.array_equal(sa[f][p], sb[f][p]), (f, p)


@pytest.mark.parametrize("name", ["28_14r", "orszag_tang"])
def test_conserved_totals(name):
    pb = PROBLEMS[name]()
    ctx, _ = run(pb, 1, 0)

    def totals():
        # level 0 everywhere (restricted under the refined level)
        s = ctx.read_state()
        l0 = [p for p, q in enumerate(pb.patches) if q[0] == 0]
        return np.array([sum(float(np.asarray(s[f][p], np.float64).sum()) for p in l0) for f in (0, 4)])

    t0 = totals()
    ctx.step(3)
    # 3 steps of FP32 updates, each rounding a cell by half an ulp: far below 1e-6 of the total
    assert np.abs(totals() - t0).max() <= 1e-6 * np.abs(t0).max()
