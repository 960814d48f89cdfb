"""The performance cases: whole calls of the library as its users make them.

Three kinds of pass:
  run      load a packed state, advance `steps` coarse steps, read the state
           back (the state stays on the device, as in a coupled program that
           exchanges it through amrmhd_set_state_all / amrmhd_get_state_all)
  adjoint  a differentiable forward and its backward through torch.autograd
  regrid   rebuild the refined levels from the state, read the state back

Sizes, patch edges, boundaries, floors and precisions are those of the
configurations, tests and benchmark of this repository, with uneven sizes
among them. Every state is a seeded analytic flow on [0, 1]^dim sampled at the
cells of each level, with a face field that is the discrete curl of a seeded
vector potential.
"""
import ctypes
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_1110_1616_gb300 import amrmhd as A
from paper_1110_1616_gb300 import inputs
from paper_1110_1616_gb300.autograd import advance as differentiable_advance

GAMMA = 5.0 / 3.0
CFL = 0.4
FLOOR = 1e-8
CLUMP_LEVELS = 6
THETA = 0.1
INFLOW = (1.0, 0.3, 0.2, 0.1, 2.5, 0.5, 0.4, 0.3)  # conserved state of the fixed inflow at x-low
WHOLE = 40_000_000  # cells up to which a level is sampled as one array


def _case(name, kind, size, psize, **more):
    size = tuple(size) + (1,) * (3 - len(size))
    c = {"kind": kind, "dim": 2 if size[2] == 1 else 3, "nx": size[0], "ny": size[1], "nz": size[2], "psize": psize,
         "levels": 1, "layout": "nested", "flow": "waves", "precision": "mixed", "steps": 1, "bounded": False,
         "floors": False, "tuned": False, "wait": False}
    c.update(more)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest 2D call: one waited-for step of the README's Orszag-Tang setup (64^2, central half refined),
        # in the default precision
        _case("amr2d_fp64_64", "run", (64, 64), 16, levels=2, precision="fp64", wait=True),
        # a production 2D run between two outputs: 512^2 with its central half refined, mixed precision
        _case("amr2d_mixed_512", "run", (512, 512), 32, levels=2, steps=4),
        # the smallest 3D call: 8 patches, far too few for the chip; latency and launches count
        _case("uniform3d_32", "run", (32, 32, 32), 16, flow="blast"),
        # the headline workload: the 128^3 blast in 512 patches of 16^3, launch shapes autotuned as the benchmark does
        _case("uniform3d_128", "run", (128, 128, 128), 16, flow="blast", steps=4, tuned=True),
        # a large uniform grid in large patches (the state is far beyond L2)
        _case("uniform3d_256", "run", (256, 256, 256), 32, flow="blast", steps=2),
        # a bounded box that patches do not tile evenly: inflow and outflow sides, floors on, ghost fills every step
        _case("bounded3d_ragged", "run", (104, 60, 76), 24, flow="waves", steps=2, bounded=True, floors=True),
        # the FP64 3D path (parity-grade runs, the default precision)
        _case("uniform3d_fp64_64", "run", (64, 64, 64), 16, flow="blast", precision="fp64"),
        # the paper's own shape: 64^3 base and one static refined level over an eighth of the volume
        _case("amr3d_two_level", "run", (64, 64, 64), 16, flow="blast", levels=2, steps=2),
        # three nested levels in patches that do not divide them
        _case("amr3d_three_level", "run", (72, 64, 56), 20, levels=3, steps=1),
        # the deep hierarchy: 6 levels of small patches around 8 clumps, 63 level advances a coarse step
        _case("clumps3d_deep", "run", (32, 32, 32), 16, layout="clumps", flow="clumps", levels=CLUMP_LEVELS, tuned=True),
        # the regrid of that hierarchy (every other coarse step in such a run)
        _case("clumps3d_regrid", "regrid", (32, 32, 32), 16, layout="clumps", flow="clumps", levels=CLUMP_LEVELS),
        # gradients of a final-state loss: 256^2 with a refined level, forward with checkpoints and backward
        _case("adjoint2d_fp64_256", "adjoint", (256, 256), 32, levels=2, precision="fp64", steps=4),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def grid(lo, hi, dim, cells, psizes):
        """Sizes of at most `cells` cells in all (multiples of 4), and a patch edge that makes at most 2000 patches."""
        size = [logint(lo, hi) // 4 * 4 for _ in range(dim)]
        while math.prod(size) > cells:
            i = size.index(max(size))
            size[i] = max(lo, size[i] // 8 * 4)
        return size, rng.choice([p for p in psizes if math.prod(-(-n // p) for n in size) <= 2000])

    kind = rng.choice(["uniform3d", "uniform3d", "nested3d", "nested3d", "fp64_3d", "two_d", "two_d", "adjoint",
                       "clumps", "regrid"])
    if kind == "uniform3d":
        size, psize = grid(16, 200, 3, 6_000_000, [8, 12, 16, 20, 24, 32])
        if rng.random() < 0.5:  # an even tiling
            size = [max(psize, v // psize * psize) for v in size]
        return _case(None, "run", size, psize, flow=rng.choice(["blast", "waves"]), steps=rng.choice([1, 2, 4]),
                     bounded=rng.random() < 0.3, floors=rng.random() < 0.25, tuned=rng.random() < 0.3,
                     wait=rng.random() < 0.3)
    if kind == "nested3d":
        size, psize = grid(24, 88, 3, 700_000, [8, 12, 16, 20, 32])
        return _case(None, "run", size, psize, flow=rng.choice(["blast", "waves"]), levels=rng.choice([2, 2, 3]),
                     steps=rng.choice([1, 2]), bounded=rng.random() < 0.25, tuned=rng.random() < 0.3,
                     wait=rng.random() < 0.3)
    if kind == "fp64_3d":
        size, psize = grid(24, 80, 3, 500_000, [8, 16, 20])
        return _case(None, "run", size, psize, flow=rng.choice(["blast", "waves"]), precision="fp64",
                     levels=rng.choice([1, 1, 2]), wait=rng.random() < 0.3)
    if kind == "two_d":
        size, psize = grid(32, 768, 2, 600_000, [8, 16, 24, 32, 64])
        return _case(None, "run", size, psize, levels=rng.choice([1, 2, 2]), precision=rng.choice(["fp64", "mixed"]),
                     steps=rng.choice([1, 2, 4]), bounded=rng.random() < 0.25, wait=rng.random() < 0.3)
    if kind == "adjoint":
        size, psize = grid(64, 256, 2, 65536, [16, 24, 32])
        return _case(None, "adjoint", size, psize, levels=rng.choice([1, 2]), precision="fp64",
                     steps=rng.choice([2, 3, 4]))
    if kind == "clumps":
        return _case(None, "run", (32, 32, 32), 16, layout="clumps", flow="clumps", levels=rng.choice([3, 4, 5, 6]),
                     steps=rng.choice([1, 2]), clumps=rng.choice([2, 4, 8]), tuned=rng.random() < 0.5)
    return _case(None, "regrid", (32, 32, 32), 16, layout="clumps", flow="clumps", levels=rng.choice([3, 4, 5, 6]),
                 clumps=rng.choice([2, 4, 8]))


# ----------------------------------------------------------------- hierarchy and state
def _base(c):
    return (c["nx"], c["ny"], c["nz"])


def _level_n(c, level):
    return [n << level if d < c["dim"] else 1 for d, n in enumerate(_base(c))]


def _clumps(c):
    return inputs.clumps_3d(base=c["nx"], nlev=c["levels"], n_clumps=c.get("clumps", 8))


def _boxes(c):
    """The region of every nested level: level 0 the domain, each finer level the central half of the one below."""
    boxes = [([0, 0, 0], _level_n(c, 0))]
    for _ in range(1, c["levels"]):
        lo, hi = boxes[-1]
        a = [2 * (lo[d] + (hi[d] - lo[d]) // 4) if d < c["dim"] else 0 for d in range(3)]
        b = [2 * (lo[d] + 3 * (hi[d] - lo[d]) // 4) if d < c["dim"] else 1 for d in range(3)]
        boxes.append((a, b))
    return boxes


def _patches(c):
    if c["layout"] == "clumps":
        return _clumps(c).patches
    out = []
    for level, (lo, hi) in enumerate(_boxes(c)):
        out += inputs.tile(level, lo, hi, c["psize"], c["dim"])
    return out


class _Flow:
    """The seeded flow: sums of a few plane waves for density, velocity, pressure and vector potential, around a
    uniform state; optionally a sphere of high pressure ("blast") or dense spheres at rest pressure ("clumps")."""

    def __init__(self, c, seed, device):
        rng = np.random.RandomState(seed % (1 << 31))
        self.c, self.device = c, device
        amp = {"waves": 0.1, "blast": 0.02, "clumps": 0.02}[c["flow"]]
        self.modes = []
        for _ in range(9):  # rho, v (3), p, A (3), B_z in 2D
            k = rng.randint(-3, 4, size=(3, 3))
            k[:, 2] *= c["dim"] - 2
            self.modes.append((k, rng.uniform(0, 2 * math.pi, 3), amp * rng.uniform(0.5, 1.0, 3) / 3))
        self.mean = {"waves": (1.0, (0.3, 0.2, 0.1), 0.8, (0.5, 0.4, 0.3)),
                     "blast": (1.0, (0.0, 0.0, 0.0), 0.1, (3 ** -0.5,) * 3),
                     "clumps": (1.0, (1.0, 0.0, 0.0), 1.0, (math.sqrt(2.0), 0.2, 0.1))}[c["flow"]]
        self.centre = 0.5 + 0.05 * rng.uniform(-1, 1, 3)
        self.spheres = _clumps(c).meta["centres"] if c["flow"] == "clumps" else []

    def wave(self, i, x, y, z):
        k, ph, a = self.modes[i]
        out = 0.0
        for m in range(3):
            out = out + a[m] * torch.sin(2 * math.pi * (k[m, 0] * x + k[m, 1] * y + k[m, 2] * z) + ph[m])
        return out

    def box(self, level, lo, hi):
        """The 8 fields on the cells [lo, hi) of a level (and on their faces), as (z, y, x) arrays."""
        n, dim = _level_n(self.c, level), self.c["dim"]
        rho0, v0, p0, b0 = self.mean

        def at(d, corner):  # coordinates along d of the cells' centres, or of their corners
            i = torch.arange(lo[d], hi[d] + (1 if corner else 0), device=self.device, dtype=torch.float64)
            if corner and not self.c["bounded"]:
                i = i % n[d]  # a periodic seam's two copies are equal bit for bit
            x = (i + (0.0 if corner else 0.5)) / n[d]
            return x.reshape([-1 if 2 - d == a else 1 for a in range(3)])

        cen = [at(d, False) for d in range(3)]
        cor = [at(d, True) for d in range(3)]
        full = [hi[2] - lo[2], hi[1] - lo[1], hi[0] - lo[0]]
        rho = (rho0 * (1 + self.wave(0, *cen))).expand(full)
        v = [(v0[d] + self.wave(1 + d, *cen)).expand(full) for d in range(3)]
        p = (p0 * (1 + self.wave(4, *cen))).expand(full)
        if self.c["flow"] == "blast":
            r2 = sum((cen[d] - self.centre[d]) ** 2 for d in range(3))
            p = torch.where(r2 < 0.01, 100 * p, p)
        for s in self.spheres:
            r2 = sum((cen[d] - float(s[d])) ** 2 for d in range(3))
            rho = torch.where(r2 < 0.02 ** 2, 100 * rho, rho)
        # B = b0 + curl A, A_e on the e-edges
        def edge(e):
            return self.wave(5 + e, *[cen[d] if d == e or d >= dim else cor[d] for d in range(3)])

        pot = [edge(e) / (2 * math.pi) if dim == 3 or e == 2 else None for e in range(3)]
        faces = []
        for d in range(dim):
            t, u = (d + 1) % 3, (d + 2) % 3
            b = torch.zeros(full[:2 - d] + [full[2 - d] + 1] + full[3 - d:], device=self.device, dtype=torch.float64)
            b += b0[d]
            if pot[u] is not None and t < dim:
                b = b + torch.diff(pot[u], dim=2 - t) * n[t]
            if pot[t] is not None and u < dim:
                b = b - torch.diff(pot[t], dim=2 - u) * n[u]
            faces.append(b)
        if dim == 2:
            faces.append((b0[2] + self.wave(8, *cen)).expand(full))
        bc = []
        for d in range(3):
            a = 2 - d
            m = faces[d].shape[a] - 1
            bc.append(0.5 * (faces[d].narrow(a, 0, m) + faces[d].narrow(a, 1, m)) if d < dim else faces[d])
        e = p / (GAMMA - 1) + 0.5 * rho * sum(x * x for x in v) + 0.5 * sum(b * b for b in bc)
        return [rho] + [rho * x for x in v] + [e] + faces


def _cut(c, fields, lo, hi):
    """The fields of the box [lo, hi) out of whole-level arrays."""
    out = []
    for f, a in enumerate(fields):
        ext = [1 if f - 5 == d and d < c["dim"] else 0 for d in range(3)]
        out.append(a[lo[2]:hi[2] + ext[2], lo[1]:hi[1] + ext[1], lo[0]:hi[0] + ext[0]])
    return out


def _packed(c, patches, level_fields):
    """The packed state: field after field, each patch after patch. level_fields[l]: whole-level arrays, or None with
    a _Flow under "flow" to sample each patch by itself."""
    parts = [[] for _ in range(8)]
    for level, lo, hi in patches:
        whole = level_fields.get(level)
        fields = _cut(c, whole, lo, hi) if whole is not None else level_fields["flow"].box(level, lo, hi)
        for f in range(8):
            parts[f].append(fields[f].reshape(-1))
    return torch.cat([torch.cat(p) for p in parts])


def _initial(c, seed, device, whole=False):
    flow = _Flow(c, seed, device)
    levels = {"flow": flow}
    for level in range(c["levels"]):
        n = _level_n(c, level)
        if whole or n[0] * n[1] * n[2] <= (WHOLE if c["layout"] != "clumps" else 300_000):
            levels[level] = flow.box(level, [0, 0, 0], n)
    return levels


def _dtype(c):
    return torch.float64 if c["precision"] == "fp64" else torch.float32


# ----------------------------------------------------------------- the cases' passes
_stream = None


def _work_stream():
    """The stream of the program: its contexts run on it one after the other."""
    global _stream
    if _stream is None:
        _stream = torch.cuda.Stream()
    return _stream


def prepare(case, seed):
    c = dict(case)
    patches = _patches(c)
    bc = [2, 1] + [1, 1] * (c["dim"] - 1) + [0, 0] * (3 - c["dim"]) if c["bounded"] else None
    cfg = A.make_config(c["dim"], _base(c)[:c["dim"]], precision=A.FP64 if c["precision"] == "fp64" else A.MIXED,
                        gamma=GAMMA, cfl=CFL, bc=bc, inflow=INFLOW if c["bounded"] else None)
    ctx = A.Context(cfg, _work_stream().cuda_stream)
    ctx.set_hierarchy(patches)
    ctx.alloc_arena()
    if c["floors"]:
        ctx.set_floors(FLOOR, FLOOR)
    levels = _initial(c, seed, "cuda")
    u = _packed(c, patches, levels)
    state = {"case": c, "ctx": ctx}
    if c["kind"] == "adjoint":
        rng = torch.Generator(device="cuda")
        rng.manual_seed(seed % (1 << 31))
        state["u0"] = u.requires_grad_(True)
        state["weight"] = torch.randn(u.numel(), device="cuda", dtype=torch.float64, generator=rng)
        state["dts"] = [0.8 * _Plain(c, levels).dt()] * c["steps"]
        state["sizes"] = [ctx.packed_size(f) for f in range(8)]
        return state
    state["u"] = u.to(_dtype(c))
    state["out"] = torch.empty_like(state["u"])
    torch.cuda.synchronize()
    if c["tuned"] or c["kind"] == "regrid":
        _exchange(state, state["u"], True)
        if c["tuned"]:
            ctx.autotune(3)
    return state


def _exchange(state, buf, into):
    """The whole packed state of the context from (into) or to a device buffer, in the context's stored type."""
    wide = buf.dtype == torch.float64
    name = ("amrmhd_set_state_all" if into else "amrmhd_get_state_all") + ("" if wide else "_f32")
    st = getattr(A.lib(), name)(state["ctx"].h, ctypes.c_void_p(buf.data_ptr()), 1)
    if st:
        raise RuntimeError("%s: status %d" % (name, st))


def run(state):
    c, ctx = state["case"], state["ctx"]
    if c["kind"] == "adjoint":
        u0 = state["u0"]
        u0.grad = None
        final = differentiable_advance(ctx, u0, state["dts"], 2)
        (final * state["weight"]).sum().backward()
        return {"final": final.detach(), "grad": list(torch.split(u0.grad, state["sizes"]))}
    if c["kind"] == "regrid":
        patches = ctx.regrid(THETA, c["levels"])
        out = torch.empty(ctx.packed_total(), dtype=_dtype(c), device="cuda")
        _exchange(state, out, False)
        return {"patches": np.array([[level, *lo, *hi] for level, lo, hi in patches], dtype=np.int32), "state": out}
    _exchange(state, state["u"], True)
    if c["wait"]:
        ctx.step(c["steps"])
    else:
        ctx.step_async(c["steps"])
    _exchange(state, state["out"], False)
    return state["out"]


def work(case):
    """One pass: every level's cells advance 2^level times a coarse step, reading and writing the 8 stored values of a
    cell once each and doing the scheme's operations (3D 1504, 2D about 900 a cell update); the packed state in and
    out once. A gradient evaluates the forward twice and its transpose, about as much again, once."""
    c = dict(case)
    size = 8 if c["precision"] == "fp64" else 4
    cells = [math.prod(hi[d] - lo[d] for d in range(3)) for _, lo, hi in _patches(c)]
    updates = sum(n << p[0] for n, p in zip(cells, _patches(c))) * c["steps"]
    per = 1504 if c["dim"] == 3 else 900
    if c["kind"] == "regrid":
        return {"bytes": 2 * 8 * size * sum(cells), "flops": 0}
    sweeps = 3 if c["kind"] == "adjoint" else 1
    return {"bytes": sweeps * updates * 16 * size + 4 * 8 * size * sum(cells), "flops": sweeps * updates * per}


# ----------------------------------------------------------------- the same results from plain torch in 64 bits
def exact(case, seed):
    c = dict(case)
    if c["kind"] == "regrid" or c["layout"] == "clumps":
        return None  # whole-level arrays of these hierarchies' finest levels (1024^3) take too long
    wide = c["kind"] == "adjoint" or c["precision"] == "fp64"
    device = "cuda" if torch.cuda.is_available() else "cpu"
    levels = _initial(c, seed, device, whole=True)
    flow = levels.pop("flow")
    if not wide:
        levels = {k: [a.float().double() for a in v] for k, v in levels.items()}
    patches = _patches(c)
    if c["kind"] == "adjoint":
        n = sum(a.numel() for a in _Plain(c, levels).packed(patches))
        rng = torch.Generator(device=device)
        rng.manual_seed(seed % (1 << 31))
        weight = torch.randn(n, device=device, dtype=torch.float64, generator=rng)
        leaves = [[a.clone().requires_grad_(True) for a in levels[k]] for k in range(c["levels"])]
        sim = _Plain(c, dict(enumerate(leaves)))
        dt = 0.8 * _Plain(c, levels).dt()
        for _ in range(c["steps"]):
            sim.checkpointed_step(dt)
        final = torch.cat(sim.packed(patches))
        (final * weight).sum().backward()
        grad = []
        for f in range(8):
            if f >= 5 and f - 5 < c["dim"]:
                grad.append(None)  # a face stored by two patches has one entry per copy: no plain value per entry
                continue
            grad.append(torch.cat([_cut(c, [a.grad for a in leaves[level]], lo, hi)[f].reshape(-1)
                                   for level, lo, hi in patches]))
        return {"final": final.detach(), "grad": grad}
    with torch.no_grad():
        sim = _Plain(c, levels)
        for _ in range(c["steps"]):
            sim.step(sim.dt())
        return torch.cat(sim.packed(patches))


def _mm(a, b):
    z = torch.zeros((), dtype=a.dtype, device=a.device)
    return torch.where((a > 0) & (b > 0), torch.where(a <= b, a, b),
                       torch.where((a < 0) & (b < 0), torch.where(a >= b, a, b), z))


class _Plain:
    """The scheme on whole-level arrays: MUSCL-Hancock with minmod slopes and a primitive predictor, HLLD fluxes,
    constrained transport with upwinded edge EMFs, subcycled levels, reflux and restriction. Face arrays keep the
    low-side face of every cell; dimensions wrap, and a bounded level 0 is padded by its ghost layers first."""

    PAD = 4

    def __init__(self, c, levels):
        self.c, self.dim, self.D = c, c["dim"], range(c["dim"])
        self.U = []
        for level in range(c["levels"]):
            n = _level_n(c, level)
            self.U.append([a if f < 5 or f - 5 >= self.dim or (c["bounded"] and level == 0)
                           else a.narrow(2 - (f - 5), 0, n[f - 5]) for f, a in enumerate(levels[level])])
        dev = self.U[0][0].device
        self.region = []
        for level, (lo, hi) in enumerate(_boxes(c)):
            n = _level_n(c, level)
            m = torch.zeros((n[2], n[1], n[0]), dtype=torch.bool, device=dev)
            m[lo[2]:hi[2], lo[1]:hi[1], lo[0]:hi[0]] = True
            self.region.append(m)

    # -- arrays
    @staticmethod
    def sh(a, d, k):
        return torch.roll(a, -k, 2 - d)

    def idx(self, level):
        return [float(_level_n(self.c, level)[d]) for d in self.D]

    def pad(self, U):
        g = self.PAD
        out = []
        for f, a in enumerate(U):
            for d in self.D:
                ax, face = 2 - d, f - 5 == d
                m = a.shape[ax]
                i = torch.arange(-g, m + g - (1 if face else 0), device=a.device)
                b = a.index_select(ax, i.clamp(0, m - 1))
                out_of = (i < 0) if d == 0 else torch.zeros_like(i, dtype=torch.bool)
                shape = [-1 if ax == e else 1 for e in range(3)]
                a = torch.where(out_of.reshape(shape), torch.full_like(b, INFLOW[f]), b)
            out.append(a)
        return out

    def crop(self, U):
        g = self.PAD
        out = []
        for f, a in enumerate(U):
            for d in self.D:
                face = f - 5 == d
                a = a.narrow(2 - d, g, a.shape[2 - d] - 2 * g + (1 if face else 0))
            out.append(a)
        return out

    def packed(self, patches):
        whole = []
        for level in range(self.c["levels"]):
            U = self.U[level]
            if not (self.c["bounded"] and level == 0):
                U = [torch.cat([a, a.narrow(2 - (f - 5), 0, 1)], 2 - (f - 5)) if f >= 5 and f - 5 < self.dim else a
                     for f, a in enumerate(U)]
            whole.append(U)
        parts = [[] for _ in range(8)]
        for level, lo, hi in patches:
            for f, a in enumerate(_cut(self.c, whole[level], lo, hi)):
                parts[f].append(a.reshape(-1))
        return [torch.cat(p) for p in parts]

    # -- the formulas of one level
    def prim(self, U):
        bc = [0.5 * (U[5 + d] + self.sh(U[5 + d], d, 1)) if d < self.dim else U[5 + d] for d in range(3)]
        v = [U[1 + d] / U[0] for d in range(3)]
        ke = 0.5 * sum(U[1 + d] * v[d] for d in range(3))
        return [U[0]] + v + [(GAMMA - 1) * (U[4] - ke - 0.5 * sum(b * b for b in bc))] + bc

    @staticmethod
    def fast2(r, p, bn, bt, bu):
        a = (GAMMA * p + bn * bn + bt * bt + bu * bu) / r
        disc = (a * a - 4 * GAMMA * p / r * (bn * bn / r)).clamp(min=0.0)
        return 0.5 * (a + torch.sqrt(disc))

    def dt(self):
        best = 0.0
        with torch.no_grad():
            for level in range(self.c["levels"]):
                U = self.U[level]
                if self.c["bounded"] and level == 0:
                    U = self.pad(U)
                w = self.prim(U)
                rate = 0.0
                for d in self.D:
                    cf = torch.sqrt(self.fast2(w[0], w[4], w[5 + d], w[5 + (d + 1) % 3], w[5 + (d + 2) % 3]))
                    rate = rate + (w[1 + d].abs() + cf) * self.idx(level)[d]
                if self.c["bounded"] and level == 0:
                    rate = self.crop([rate])[0]
                best = max(best, float(rate[self.region[level]].max()) * 0.5 ** level)
        return CFL / best

    @staticmethod
    def hlld(ql, qr, bn):
        def flux(q):
            r, un, ut, uu, p, bt, bu = q
            b2 = bn * bn + bt * bt + bu * bu
            pt = p + 0.5 * b2
            e = p / (GAMMA - 1) + 0.5 * r * (un * un + ut * ut + uu * uu) + 0.5 * b2
            vb = un * bn + ut * bt + uu * bu
            return ([r * un, r * un * un + pt - bn * bn, r * un * ut - bn * bt, r * un * uu - bn * bu,
                     (e + pt) * un - bn * vb, bt * un - bn * ut, bu * un - bn * uu],
                    [r, r * un, r * ut, r * uu, e, bt, bu], pt)

        fl, ul, ptl = flux(ql)
        fr, ur, ptr = flux(qr)
        c = torch.sqrt(torch.maximum(_Plain.fast2(ql[0], ql[4], bn, ql[5], ql[6]),
                                     _Plain.fast2(qr[0], qr[4], bn, qr[5], qr[6])))
        sl, sr = torch.minimum(ql[1], qr[1]) - c, torch.maximum(ql[1], qr[1]) + c
        dl, dr = (sl - ql[1]) * ql[0], (sr - qr[1]) * qr[0]
        den = dr - dl
        sm = (dr * qr[1] - dl * ql[1] - ptr + ptl) / den
        pts = (dr * ptl - dl * ptr + dr * dl * (qr[1] - ql[1])) / den
        bn2 = bn * bn
        star = []
        for q, u, s, pt in ((ql, ul, sl, ptl), (qr, ur, sr, ptr)):
            da, ssm = s - q[1], s - sm
            rs = q[0] * da / ssm
            e = q[0] * da * ssm - bn2
            flat = e.abs() <= 1e-12 * ((e + bn2).abs() + bn2)
            ie = 1.0 / torch.where(flat, torch.ones_like(e), e)
            tq, qq = bn * (sm - q[1]) * ie, (q[0] * da * da - bn2) * ie
            vs = torch.where(flat, q[2], q[2] - q[5] * tq)
            ws = torch.where(flat, q[3], q[3] - q[6] * tq)
            bt = torch.where(flat, q[5], q[5] * qq)
            bu = torch.where(flat, q[6], q[6] * qq)
            vb = q[1] * bn + q[2] * q[5] + q[3] * q[6]
            vbs = sm * bn + vs * bt + ws * bu
            es = (da * u[4] - pt * q[1] + pts * sm + bn * (vb - vbs)) / ssm
            star.append((rs, vs, ws, bt, bu, es, vbs, [rs, rs * sm, rs * vs, rs * ws, es, bt, bu]))
        (rl, vl, wl, btl, bul, el, vbl, usl), (rr, vr, wr, btr, bur, er, vbr, usr) = star
        ok = (rl > 0) & (rr > 0)
        one = torch.ones_like(rl)
        sql, sqr = torch.sqrt(torch.where(ok, rl, one)), torch.sqrt(torch.where(ok, rr, one))
        sls, srs = sm - bn.abs() / sql, sm + bn.abs() / sqr
        sg = torch.where(bn > 0, one, -one)
        i = 1.0 / (sql + sqr)
        vss = (sql * vl + sqr * vr + (btr - btl) * sg) * i
        wss = (sql * wl + sqr * wr + (bur - bul) * sg) * i
        bts = (sql * btr + sqr * btl + sql * sqr * (vr - vl) * sg) * i
        bus = (sql * bur + sqr * bul + sql * sqr * (wr - wl) * sg) * i
        vbs = sm * bn + vss * bts + wss * bus
        ell, err = el - sql * (vbl - vbs) * sg, er + sqr * (vbr - vbs) * sg
        dl = [rl, rl * sm, rl * vss, rl * wss, ell, bts, bus]
        dr = [rr, rr * sm, rr * vss, rr * wss, err, bts, bus]
        single = bn2 <= 1e-12 * pts
        left = sm >= 0
        out = []
        for k in range(7):
            f1l, f1r = fl[k] + sl * (usl[k] - ul[k]), fr[k] + sr * (usr[k] - ur[k])
            f2l = fl[k] + sls * dl[k] - (sls - sl) * usl[k] - sl * ul[k]
            f2r = fr[k] + srs * dr[k] - (srs - sr) * usr[k] - sr * ur[k]
            f = torch.where(left, f2l, f2r)
            f = torch.where(srs <= 0, f1r, f)
            f = torch.where(sls >= 0, f1l, f)
            f = torch.where(single, torch.where(left, f1l, f1r), f)
            f = torch.where(sr < 0, fr[k], f)
            out.append(torch.where(sl > 0, fl[k], f))
        return out

    def advance(self, U, level, dt):
        """(new state, fluxes by direction and field, EMFs by component) of one advance of a whole level."""
        sh, dim = self.sh, self.dim
        idx = self.idx(level)
        w = self.prim(U)
        slope = [[sh(U[5 + d], d, 1) - U[5 + d] if f == 5 + d else _mm(w[f] - sh(w[f], d, -1), sh(w[f], d, 1) - w[f])
                  for f in range(8)] for d in self.D]
        wh = list(w)
        for d in self.D:
            n, t, u = d, (d + 1) % 3, (d + 2) % 3
            s, vn, bn, bt, bu = slope[d], w[1 + n], w[5 + n], w[5 + t], w[5 + u]
            dw = [None] * 8
            dw[0] = vn * s[0] + w[0] * s[1 + n]
            dw[1 + n] = vn * s[1 + n] + (s[4] + bt * s[5 + t] + bu * s[5 + u]) / w[0]
            dw[1 + t] = vn * s[1 + t] - bn * s[5 + t] / w[0]
            dw[1 + u] = vn * s[1 + u] - bn * s[5 + u] / w[0]
            dw[4] = vn * s[4] + GAMMA * w[4] * s[1 + n]
            dw[5 + n] = vn * s[5 + n]
            dw[5 + t] = vn * s[5 + t] - bn * s[1 + t] + bt * s[1 + n]
            dw[5 + u] = vn * s[5 + u] - bn * s[1 + u] + bu * s[1 + n]
            wh = [a - 0.5 * dt * idx[d] * b for a, b in zip(wh, dw)]
        ref = [wh[3] * wh[6] - wh[2] * wh[7], wh[1] * wh[7] - wh[3] * wh[5], wh[2] * wh[5] - wh[1] * wh[6]]
        F = []
        for d in self.D:
            n, t, u = d, (d + 1) % 3, (d + 2) % 3
            left = [sh(a + 0.5 * s, d, -1) for a, s in zip(wh, slope[d])]
            right = [a - 0.5 * s for a, s in zip(wh, slope[d])]
            order = [0, 1 + n, 1 + t, 1 + u, 4, 5 + t, 5 + u]
            f = self.hlld([left[k] for k in order], [right[k] for k in order], 0.5 * (left[5 + n] + right[5 + n]))
            g = [None] * 8
            for k, o in enumerate(order):
                g[o] = f[k]
            F.append(g)
        E = [None] * 3
        for e in ((2,) if dim == 2 else (0, 1, 2)):
            a, b = (e + 1) % 3, (e + 2) % 3
            up = lambda m, lo, hi: torch.where(m > 0, lo, torch.where(m < 0, hi, 0.5 * (lo + hi)))  # noqa: E731
            ea, eb = -F[a][5 + b], F[b][5 + a]
            ea_lo, eb_lo = sh(ea, b, -1), sh(eb, a, -1)
            # cells around the edge by their offsets along (a, b)
            r11, r01, r10 = ref[e], sh(ref[e], a, -1), sh(ref[e], b, -1)
            r00 = sh(r10, a, -1)
            ma, mb = F[a][0], F[b][0]
            db_hi = up(ma, r01 - eb_lo, r11 - eb)
            db_lo = up(sh(ma, b, -1), eb_lo - r00, eb - r10)
            da_hi = up(mb, r10 - ea_lo, r11 - ea)
            da_lo = up(sh(mb, a, -1), ea_lo - r00, ea - r01)
            E[e] = 0.25 * (ea + ea_lo + eb + eb_lo) + 0.25 * (db_lo - db_hi) + 0.25 * (da_lo - da_hi)
        V = []
        for f in range(8):
            v = U[f]
            if f < 5 or f - 5 >= dim:
                for d in self.D:
                    v = v - dt * idx[d] * (sh(F[d][f], d, 1) - F[d][f])
            else:
                v = v + dt * self.curl(E, f - 5, idx)
            V.append(v)
        return V, F, E

    def curl(self, E, d, idx):
        t, u = (d + 1) % 3, (d + 2) % 3
        out = 0.0
        if E[u] is not None and t < self.dim:
            out = out - idx[t] * (self.sh(E[u], t, 1) - E[u])
        if E[t] is not None and u < self.dim:
            out = out + idx[u] * (self.sh(E[t], u, 1) - E[t])
        return out

    # -- between levels
    def up(self, a):
        for d in self.D:
            a = a.repeat_interleave(2, 2 - d)
        return a

    def sign(self, a, d):
        s = torch.tensor([-0.25, 0.25], dtype=a.dtype, device=a.device).repeat(a.shape[2 - d] // 2)
        return s.reshape([-1 if 2 - d == e else 1 for e in range(3)])

    def slope(self, a, d):
        return _mm(a - self.sh(a, d, -1), self.sh(a, d, 1) - a)

    def prolong(self, U):
        out = []
        for f in range(8):
            n = f - 5
            if f < 5 or n >= self.dim:
                v = self.up(U[f])
                out.append(v + sum(self.up(self.slope(U[f], d)) * self.sign(v, d) for d in self.D))
                continue
            lo = self.up(U[f])
            lo = lo + sum(self.up(self.slope(U[f], d)) * self.sign(lo, d) for d in self.D if d != n)
            hi = self.sh(lo, n, 2)  # the coarse cell's high face, at the same transverse children
            corr = 0.0
            ratio = [1.0 / x for x in self.idx(0)]
            for t in self.D:
                if t != n:
                    s = self.slope(U[5 + t], n)
                    corr = corr + ratio[n] / ratio[t] * (self.sh(s, t, 1) - s)
            mid = 0.5 * (lo + hi) + 0.125 * self.up(corr)
            i = torch.arange(lo.shape[2 - n], device=lo.device).reshape([-1 if 2 - n == e else 1 for e in range(3)])
            out.append(torch.where(i % 2 == 0, lo, mid))
        return out

    def down(self, a, dims):
        """The mean over the children along `dims`, at the low child along the other dimensions."""
        for d in self.D:
            b = a.unflatten(2 - d, (-1, 2))
            a = b.mean(2 - d + 1) if d in dims else b.select(2 - d + 1, 0)
        return a

    def faces_of(self, mask, d):
        return mask | self.sh(mask, d, -1)

    def fill(self, level, coarse):
        P = self.prolong(coarse)
        r = self.region[level]
        self.U[level] = [torch.where(r if f < 5 or f - 5 >= self.dim else self.faces_of(r, f - 5), a, b)
                         for f, (a, b) in enumerate(zip(self.U[level], P))]

    def covered(self, level):
        m = self.region[level + 1]
        for d in self.D:
            m = m.unflatten(2 - d, (-1, 2)).select(2 - d + 1, 0)
        return m

    def sub_step(self, level, dt):
        """One advance of a level and of everything finer; returns its fluxes and EMFs for the registers."""
        padded = self.c["bounded"] and level == 0
        before = self.pad(self.U[level]) if padded else self.U[level]
        V, F, E = self.advance(before, level, dt)
        if padded:
            V = self.crop(V)
            g = self.PAD
            cut = lambda a: None if a is None else a[tuple(slice(g, -g) if 2 - e in self.D else slice(None) for e in range(3))]  # noqa: E731
            before = [cut(a) for a in before]
            F, E = [[cut(a) for a in f] for f in F], [cut(a) for a in E]
        self.U[level] = V
        if level + 1 < self.c["levels"]:
            self.fill(level + 1, before)
            Fs, Es = [], []
            for _ in range(2):
                f, e = self.sub_step(level + 1, 0.5 * dt)
                Fs.append(f)
                Es.append(e)
            self.synchronise(level, dt, F, E, Fs, Es)
        return F, E

    def synchronise(self, level, dt, F, E, Fs, Es):
        cov, idx, dim, sh = self.covered(level), self.idx(level), self.dim, self.sh
        U, V = list(self.U[level]), self.U[level + 1]
        padded = self.c["bounded"] and level == 0
        low = lambda f: U[f].narrow(2 - (f - 5), 0, cov.shape[2 - (f - 5)]) if padded else U[f]  # noqa: E731
        for f in range(8):
            if f >= 5 and f - 5 < dim:
                continue
            for d in self.D:
                across = [t for t in self.D if t != d]
                R = 0.5 * dt * (self.down(Fs[0][d][f], across) + self.down(Fs[1][d][f], across)) - dt * F[d][f]
                R = torch.where(cov ^ sh(cov, d, -1), R, torch.zeros_like(R))
                U[f] = U[f] + torch.where(cov, torch.zeros_like(R), idx[d] * (R - sh(R, d, 1)))
        RE = [None] * 3
        for e in range(3):
            if E[e] is None:
                continue
            along = [e] if e < dim else []
            a, b = (e + 1) % 3, (e + 2) % 3
            k = sum(m.int() for m in (cov, sh(cov, a, -1), sh(cov, b, -1), sh(sh(cov, a, -1), b, -1)))
            R = 0.5 * dt * (self.down(Es[0][e], along) + self.down(Es[1][e], along)) - dt * E[e]
            RE[e] = torch.where((k > 0) & (k < 4), R, torch.zeros_like(R))
        for d in self.D:
            free = ~cov & ~sh(cov, d, -1)
            f = 5 + d
            b = low(f)
            b = torch.where(free, b + self.curl(RE, d, idx), b)
            b = torch.where(self.faces_of(cov, d), self.down(V[f], [t for t in self.D if t != d]), b)
            if padded:
                b = torch.cat([b, U[f].narrow(2 - d, cov.shape[2 - d], 1)], 2 - d)
            U[f] = b
        for f in range(8):
            if f < 5 or f - 5 >= dim:
                U[f] = torch.where(cov, self.down(V[f], list(self.D)), U[f])
        self.U[level] = U

    def step(self, dt):
        self.sub_step(0, dt)

    def checkpointed_step(self, dt):
        """step() kept differentiable with only its input and output stored."""
        shape = [len(u) for u in self.U]

        def body(*flat):
            flat = list(flat)
            self.U = [[flat.pop(0) for _ in range(k)] for k in shape]
            self.step(dt)
            return tuple(a for u in self.U for a in u)

        flat = torch.utils.checkpoint.checkpoint(body, *[a for u in self.U for a in u], use_reentrant=False)
        flat = list(flat)
        self.U = [[flat.pop(0) for _ in range(k)] for k in shape]
