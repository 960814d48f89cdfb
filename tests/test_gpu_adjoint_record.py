"""A recorded forward ends where a later call replaces the memory it lives in,
also when that call then fails for want of memory: amrmhd_backward_recorded
answers AMRMHD_ESTATE (no record), and the next recorded forward and its backward
are what they were. The failure is an allocation no GPU can serve (terabytes),
which the driver refuses at once."""
import numpy as np
import pytest

from helpers import levels_to_packed_seed, oracle_for
from paper_1110_1616_gb300 import amrmhd as A
from test_gpu_adjoint import PROBLEMS, built, quadrant_2d, gpu_ctx, random_lam, stored_mask  # noqa: F401

pytestmark = pytest.mark.gpu
MANY = 1 << 24


# snapshots of all steps at once; checkpoints every 2 and (after larger snapshots were had) every 3 steps
@pytest.mark.parametrize("call", ["backward", "step_dt_ckpt"])
@pytest.mark.parametrize("ckpt", [MANY, 2, 3])
def test_no_record_after_its_memory_was_lost(call, ckpt):
    import torch
    pb = PROBLEMS["quadrant_2d"]()
    o = oracle_for(pb)
    dts = [o.step() for _ in range(4)]
    ctx = gpu_ctx(pb)
    seed = torch.tensor(levels_to_packed_seed(ctx, pb, random_lam(pb, np.random.default_rng(7), stored_mask(ctx, pb))),
                        dtype=torch.float64, device="cuda")
    u0, g, ref = (torch.empty_like(seed) for _ in range(3))
    torch.cuda.synchronize()
    ctx.read_packed_all(u0)
    ctx.backward(dts, seed, ref, 2)
    ctx.step_dt_ckpt(dts, 2)
    with pytest.raises(A.AmrmhdError) as e:
        many = np.full(MANY, dts[0])
        ctx.backward(many, seed, g, ckpt) if call == "backward" else ctx.step_dt_ckpt(many, ckpt)
    assert e.value.status == A.ECUDA
    assert not ctx.backward_recorded(seed, g)
    ctx.load_packed_all(u0)
    ctx.step_dt_ckpt(dts, 2)
    assert ctx.backward_recorded(seed, g)
    # the order of the atomic FP64 additions varies from run to run
    assert (g - ref).abs().max() <= 1e-12 * ref.abs().max()


def test_a_lower_limit_gives_the_kept_stages_back():
    """AMRMHD_OPT_ADJOINT_KEEP set below what is held returns the memory at once, and the record's gradient stays."""
    import torch
    pb = quadrant_2d(64)
    o = oracle_for(pb)
    dts = [o.step() for _ in range(4)]
    ctx = gpu_ctx(pb)
    seed = torch.tensor(levels_to_packed_seed(ctx, pb, random_lam(pb, np.random.default_rng(9), stored_mask(ctx, pb))),
                        dtype=torch.float64, device="cuda")
    u0, g, ref = (torch.empty_like(seed) for _ in range(3))
    torch.cuda.synchronize()
    ctx.read_packed_all(u0)
    ctx.set_option(A.OPT_ADJOINT_KEEP, 0)
    ctx.backward(dts, seed, ref, 4)

    def free():
        torch.cuda.synchronize()
        return torch.cuda.mem_get_info()[0]

    assert (ref - ref).abs().max() <= 1e-12 * ref.abs().max()  # the comparison's own memory is taken from here on
    none = free()
    ctx.set_option(A.OPT_ADJOINT_KEEP, -1)
    ctx.step_dt_ckpt(dts, 4)
    held = none - free()
    # 70 stage arrays a cell at least, for the coarse and twice the refined level's cells of 4 steps
    least = 4 * 70 * 8 * 3 * 64 * 64
    assert held >= least
    for limit in (least // 8, 0):
        ctx.set_option(A.OPT_ADJOINT_KEEP, limit)
        assert none - free() <= limit
        assert ctx.backward_recorded(seed, g)
        assert (g - ref).abs().max() <= 1e-12 * ref.abs().max()
        ctx.load_packed_all(u0)
        ctx.step_dt_ckpt(dts, 4)
        assert none - free() <= limit + (2 << 20)  # an allocation is rounded up


def test_a_workspace_that_did_not_fit_is_not_used():
    """The adjoint's first call fails while something else holds the device memory, and works once that is gone."""
    import torch
    pb = quadrant_2d(128)
    o = oracle_for(pb)
    dts = [o.step() for _ in range(2)]
    ctx = gpu_ctx(pb)
    seed = torch.tensor(levels_to_packed_seed(ctx, pb, random_lam(pb, np.random.default_rng(3), stored_mask(ctx, pb))),
                        dtype=torch.float64, device="cuda")
    g, ref = torch.empty_like(seed), torch.empty_like(seed)
    ctx.fill_ghosts(0, 1)  # the context's own lazy memory
    torch.cuda.synchronize()
    # the adjoint's scratch of every cell is 2 x 70 values: leave room for less than half of it
    need = 2 * 70 * 8 * 2 * 128 * 128
    rest = torch.empty(torch.cuda.mem_get_info()[0] - need // 2, dtype=torch.uint8, device="cuda")
    for _ in range(2):
        with pytest.raises(A.AmrmhdError) as e:
            ctx.backward(dts, seed, ref, 2)
        assert e.value.status == A.ECUDA
    del rest
    torch.cuda.empty_cache()
    ctx.backward(dts, seed, ref, 2)
    ctx.step_dt_ckpt(dts, 2)
    assert ctx.backward_recorded(seed, g)
    assert (g - ref).abs().max() <= 1e-12 * ref.abs().max()
