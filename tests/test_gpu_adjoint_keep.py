"""The adjoint's kept stage arrays (AMRMHD_OPT_ADJOINT_KEEP): the recorded
forward's gradient with none, some and all steps of a segment kept equals the
gradient with everything recomputed, and the two sides agree when the option
changes between them.

FP64 (in mixed precision the seeds of the local Jacobians are rounded to FP32,
so two runs of one call differ by an FP32 rounding here and there). Tolerance:
the stage arrays are the same bits kept or recomputed; only the
order of the adjoint's atomic FP64 additions varies from run to run: 1e-12 of
the largest gradient entry, as for the checkpoint interval.
"""
import numpy as np
import pytest

from helpers import levels_to_packed_seed, oracle_for
from paper_1110_1616_gb300 import amrmhd as A
from test_gpu_adjoint import PROBLEMS, built, gpu_ctx, random_lam, stored_mask  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,ckpt", [("quadrant_2d", 2), ("three_level_2d", 3), ("bounded_2d", 5), ("small_3d", 4)])
def test_kept_stages_do_not_change_the_gradient(name, ckpt):
    import torch
    pb = PROBLEMS[name]()
    o = oracle_for(pb)
    dts = [o.step() for _ in range(5)]
    ctx = gpu_ctx(pb)
    seed = torch.tensor(levels_to_packed_seed(ctx, pb, random_lam(pb, np.random.default_rng(5), stored_mask(ctx, pb))),
                        dtype=torch.float64, device="cuda")
    g = torch.empty_like(seed)
    torch.cuda.synchronize()
    ctx.set_option(A.OPT_ADJOINT_KEEP, 0)
    ctx.backward(dts, seed, g, ckpt)
    ref = g.cpu().numpy()
    # a state's elements x 70 / 8 fields is a level's stage arrays: room for a step or two, then for all
    some = int(ctx.packed_total() * 70 / 8 * 8 * 2 ** len(pb.state) * 2)
    for keep in (some, -1, 0):
        ctx.set_option(A.OPT_ADJOINT_KEEP, keep)
        ctx.step_dt_ckpt(dts, ckpt)
        ctx.set_option(A.OPT_ADJOINT_KEEP, -1)
        assert ctx.backward_recorded(seed, g)
        assert np.abs(g.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
        ctx.set_option(A.OPT_ADJOINT_KEEP, keep)
        ctx.backward(dts, seed, g, ckpt)
        assert np.abs(g.cpu().numpy() - ref).max() <= 1e-12 * np.abs(ref).max()
