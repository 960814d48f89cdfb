"""The FP64 CFL reduction where a cell's two face fields nearly cancel, so that
their mean is far smaller than what 24 bits of them resolve: dt still equals, bit
for bit, the oracle's over all cells, and a cell whose pressure is not positive
is still reported."""
import numpy as np
import pytest

from helpers import oracle_for
from paper_1110_1616_gb300 import amrmhd as A
from paper_1110_1616_gb300 import inputs
from test_gpu_cfl_pruned import built, context  # noqa: F401

pytestmark = pytest.mark.gpu


def problem(dim, n, faces, seed, spread):
    """Cells of O(1) pressure and field between faces of alternating sign and magnitude `faces`."""
    rng = np.random.default_rng(seed)
    nz = n if dim == 3 else 1
    c = (nz, n, n)
    rho = np.exp(0.1 * spread * rng.normal(size=c))
    p = np.exp(0.1 * spread * rng.normal(size=c))
    v = [spread * rng.normal(size=c) for _ in range(3)]
    field, cell = [], []
    for d in range(3):
        ax = 2 - d
        if d >= dim:
            field.append(rng.normal(size=c))
            cell.append(field[-1])
            continue
        shape = [m + (a == ax) for a, m in enumerate(c)]
        i = np.arange(n + 1).reshape([-1 if a == ax else 1 for a in range(3)])
        f = np.where(i % 2 == 0, faces, -faces) + spread * rng.normal(size=shape)
        np.moveaxis(f, ax, 0)[n] = np.moveaxis(f, ax, 0)[0]  # the periodic seam (n is even)
        field.append(f)
        cell.append(0.5 * (np.take(f, range(n), axis=ax) + np.take(f, range(1, n + 1), axis=ax)))
    e = p / (inputs.GAMMA - 1) + 0.5 * rho * sum(x * x for x in v) + 0.5 * sum(x * x for x in cell)
    base = (n, n, nz)
    return inputs.Problem("cancel", dim, base, inputs.tile(0, (0, 0, 0), base, 16, dim), 1,
                          {0: [rho, rho * v[0], rho * v[1], rho * v[2], e] + field})


@pytest.mark.parametrize("faces", [1.0, 3e1, 1e3, 1e5, 1e7])
@pytest.mark.parametrize("dim,n", [(2, 192), (3, 48)])
@pytest.mark.parametrize("spread", [1.0, 1e-4])
def test_dt_equals_the_oracle_bitwise(dim, n, faces, spread):
    for seed in range(3):
        pb = problem(dim, n, faces, seed, spread)
        assert context(pb).cfl_dt() == oracle_for(pb).cfl_dt()


@pytest.mark.parametrize("faces,mean", [(190.0, 2.28e-5), (190.0, 1.1e-5), (1e4, 5e-4)])
def test_a_cell_without_pressure_behind_cancelling_faces_is_reported(faces, mean):
    pb = problem(3, 48, 0.5, 4, 0.1)
    st = pb.state[0]
    z, y, x = 9, 21, 30
    for f in (1, 2, 3):
        st[f][z, y, x] = 0.0
    st[0][z, y, x] = 1.0
    for d in range(3):
        lo, hi = [z, y, x], [z, y, x]
        hi[2 - d] += 1
        st[5 + d][tuple(lo)], st[5 + d][tuple(hi)] = (faces + 2 * mean, -faces) if d == 0 else (0.0, 0.0)
    # the cells around it share its faces: their energies follow
    bc = [0.5 * (np.take(st[5 + d], range(48), 2 - d) + np.take(st[5 + d], range(1, 49), 2 - d)) for d in range(3)]
    st[4][:] = 1.5 + 0.5 * sum(st[f] ** 2 for f in (1, 2, 3)) / st[0] + 0.5 * sum(b * b for b in bc)
    assert context(pb).cfl_dt() == oracle_for(pb).cfl_dt()
    st[4][z, y, x] = 0.5 * bc[0][z, y, x] ** 2 * (1 - 1e-3)
    with pytest.raises(A.AmrmhdError) as e:
        context(pb).cfl_dt()
    assert e.value.status == A.ENONPHYS
