"""The mixed path's results bit for bit: check sums of the state and of the time
steps after a few coarse steps, recorded from the formulas as they are written
(hlld_plain, the energy balance and the restriction in FP64) before the FP32
kernels restated them. The rounding decides the sign of the mass flux of gas
nearly at rest and with it what the edge EMFs upwind, so a restated formula of
the same accuracy moves single faces by far more than a rounding; and the
results must not depend on the tile or the split of the columns. Inputs from
integers and the four basic operations only, so that they are the same bits
everywhere."""
import math
import zlib

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


def _tri(seed, n, dim, at):
    """A triangular wave in [-1/2, 1/2] over integer positions (n periods of which fit the domain)."""
    r = np.random.default_rng(seed).integers(0, 1 << 20, 4)
    t = sum(int(r[d] % 3 + 1) * at[d] for d in range(dim)) + int(r[3] % n)
    return np.abs(2 * (t % n) - n) / n - 0.5


def _level(n, dim):
    """The 8 fields of a level of n cells a side: half of the gas at rest, a box of high pressure."""
    shape = (n[2], n[1], n[0])

    def at(half):  # cell centres or corners along each direction, in half cells
        return [(2 * np.arange(n[d] + (d in half)) + (d not in half)).reshape([-1 if a == 2 - d else 1 for a in range(3)])
                for d in range(3)]

    N = 2 * math.gcd(*n[:dim])  # periodic in every direction
    N = N if N >= 32 else 2 * n[0]
    cen = at(())
    full = np.zeros(shape)
    rho = 1.0 + 0.25 * _tri(1, N, dim, cen) + full
    move = cen[0] >= n[0]
    v = [np.where(move, 0.25 + 0.25 * _tri(2 + d, N, dim, cen), 0.0) + full for d in range(3)]
    box = np.ones((1, 1, 1), bool)
    for d in range(dim):
        box = box & (np.abs(cen[d] - n[d]) * 4 < n[d])
    p = np.where(box, 12.0, 0.75) + 0.25 * _tri(5, N, dim, cen) + full
    b0 = (0.5, 0.25, 0.125)
    pot = [_tri(6 + e, N, dim, at([d for d in range(dim) if d != e])) / 32.0 for e in range(3)]
    faces = []
    for d in range(3):
        if d >= dim:
            faces.append(b0[d] + 0.125 * _tri(9, N, dim, cen) + full)
            continue
        t, u = (d + 1) % 3, (d + 2) % 3
        f = np.zeros([n[2 - a] + (a == 2 - d) for a in range(3)]) + b0[d]
        if t < dim:
            f = f + np.diff(pot[u] + np.zeros([n[2 - a] + (a == 2 - d or a == 2 - t) for a in range(3)]), axis=2 - t)
        if u < dim:
            f = f - np.diff(pot[t] + np.zeros([n[2 - a] + (a == 2 - d or a == 2 - u) for a in range(3)]), axis=2 - u)
        faces.append(f)
    bc = []
    for d in range(3):
        a, m = 2 - d, faces[d].shape[2 - d]
        bc.append(faces[d] if d >= dim else 0.5 * (np.take(faces[d], range(m - 1), a) + np.take(faces[d], range(1, m), a)))
    e = p / (inputs.GAMMA - 1.0) + 0.5 * rho * (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]) + \
        0.5 * (bc[0] * bc[0] + bc[1] * bc[1] + bc[2] * bc[2])
    return [rho] + [rho * x for x in v] + [e] + faces


def _problem(base, psize, nlev, bounded):
    dim = 2 if base[2] == 1 else 3
    patches = inputs.tile(0, (0, 0, 0), base, psize, dim)
    if nlev == 2:
        patches += inputs.tile(1, tuple(base[d] // 2 if d < dim else 0 for d in range(3)),
                               tuple(3 * base[d] // 2 if d < dim else 1 for d in range(3)), psize, dim)
    state = {lev: _level([base[d] << lev if d < dim else 1 for d in range(3)], dim) for lev in range(nlev)}
    bc = (2, 1) + (1, 1) * (dim - 1) + (0, 0) * (3 - dim) if bounded else None
    return inputs.Problem("bits", dim, base, patches, nlev, state, bc=bc,
                          inflow=(1.0, 0.25, 0.125, 0.0, 2.5, 0.5, 0.25, 0.125) if bounded else None)


# base, patch edge, levels, physical boundaries with floors, coarse steps
CASES = {"uniform": ((32, 32, 32), 16, 1, False, 4), "ragged": ((36, 28, 20), 16, 1, True, 3),
         "large": ((96, 64, 64), 32, 1, False, 3), "two_level": ((32, 48, 32), 16, 2, False, 3),
         "two_level_20": ((40, 40, 40), 20, 2, False, 2),
         "bounded_two_level": ((32, 32, 40), 20, 2, True, 2),
         "2d": ((96, 64, 1), 16, 1, False, 4), "2d_two_level": ((64, 64, 1), 32, 2, False, 4)}
RECORDED = {"uniform": "5dcfdcfc", "ragged": "4831eaf0", "large": "6f761f38", "two_level": "36801d5a",
            "two_level_20": "295c6fb1", "bounded_two_level": "76c769e1",
            "2d": "84cd08e6", "2d_two_level": "aba44d16"}


def context(name, tile=-1, zchunk=-1, advance=0, bad=None):
    import torch
    base, psize, nlev, bounded, steps = CASES[name]
    pb = _problem(base, psize, nlev, bounded)
    cfg = A.make_config(pb.dim, pb.base, precision=A.MIXED, gamma=pb.gamma, cfl=pb.cfl, bc=pb.bc, inflow=pb.inflow)
    ctx = A.Context(cfg, torch.cuda.Stream().cuda_stream)
    for option, value in ((A.OPT_ADVANCE, advance), (A.OPT_TILE, tile), (A.OPT_ZCHUNK, zchunk)):
        ctx.set_option(option, value)
    ctx.set_hierarchy(pb.patches)
    ctx.alloc_arena()
    if bounded:
        ctx.set_floors(1e-8, 1e-8)
    torch.cuda.synchronize()
    if bad is not None:  # a field and its value in one cell of level 0
        pb.state[0][bad[0]][(0 if pb.dim == 2 else 5), 9, 11] = bad[1]
    ctx.load_state(pb.state)
    return ctx, steps


def check(ctx, dts, finite=True):
    out = [zlib.crc32(dts.tobytes())]
    for f in range(8):
        x = ctx.get_field_packed(f).astype(np.float32) + np.float32(0.0)  # one zero
        assert not finite or np.isfinite(x).all()
        x[np.isnan(x)] = np.nan  # one NaN
        out.append(zlib.crc32(x.tobytes()))
    return "%08x" % zlib.crc32(np.array(out, np.uint64).tobytes())


def sums(name, tile=-1, zchunk=-1, advance=0):
    ctx, steps = context(name, tile, zchunk, advance)
    return check(ctx, ctx.step(steps))


@pytest.mark.parametrize("name", list(CASES))
def test_recorded_bits(name):
    assert sums(name) == RECORDED[name]


@pytest.mark.parametrize("tile", range(5))
@pytest.mark.parametrize("name", ["uniform", "ragged", "two_level_20"])
def test_every_launch_shape_gives_the_recorded_bits(name, tile):
    assert sums(name, tile, 0) == RECORDED[name]
    assert sums(name, tile, 5) == RECORDED[name]


@pytest.mark.parametrize("name", ["2d", "2d_two_level"])
def test_the_staged_2d_kernels_give_the_recorded_bits(name):
    assert sums(name, advance=2) == RECORDED[name]


@pytest.mark.parametrize("name", ["2d", "2d_two_level", "uniform", "two_level"])
def test_steps_of_given_dt_are_the_same_run(name):
    """What amrmhd_step_dt advances (and the adjoint differentiates) is the run that amrmhd_step makes."""
    ctx, steps = context(name)
    dts = ctx.step(steps)
    again, _ = context(name)
    again.step_dt(dts)
    assert check(again, dts) == RECORDED[name]


# density or energy of one cell, and the check sums after two steps of a given dt
BAD = {"rho_nan": (0, np.nan), "rho_0": (0, 0.0), "rho_negative": (0, -1.0), "E_nan": (4, np.nan), "E_inf": (4, np.inf),
       "E_0": (4, 0.0), "m_inf": (1, -np.inf)}
RECORDED_BAD = {
    ("uniform", "rho_nan"): "fcd028fa", ("uniform", "rho_0"): "c7c1a865", ("uniform", "rho_negative"): "4435255d",
    ("uniform", "E_nan"): "4dea2d44", ("uniform", "E_inf"): "bf82c4bc", ("uniform", "E_0"): "c14d635e",
    ("uniform", "m_inf"): "4dea2d44",
    ("ragged", "rho_nan"): "ef3ce89d", ("ragged", "rho_0"): "f1ccc5bd", ("ragged", "rho_negative"): "9551409b",
    ("ragged", "E_nan"): "74de804a", ("ragged", "E_inf"): "0ca87bb5", ("ragged", "E_0"): "b07c8e3e",
    ("ragged", "m_inf"): "74de804a",
    ("2d", "rho_nan"): "0bac42bd", ("2d", "rho_0"): "b4905d10", ("2d", "rho_negative"): "6eccb5a0",
    ("2d", "E_nan"): "30b083b0", ("2d", "E_inf"): "30b083b0", ("2d", "E_0"): "522943fc",
    ("2d", "m_inf"): "58fa2120",
}


@pytest.mark.parametrize("bad", list(BAD))
@pytest.mark.parametrize("name", ["uniform", "ragged", "2d"])
def test_a_cell_that_is_no_gas_spreads_as_recorded(name, bad):
    """amrmhd_step_dt does not look at the state: what a broken cell does to the others is fixed too."""
    ctx, _ = context(name, bad=BAD[bad])
    dts = np.array([0.001, 0.0015])
    ctx.step_dt(dts)
    assert check(ctx, dts, False) == RECORDED_BAD[name, bad]
