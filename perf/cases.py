"""Workloads of the library as a user's program runs them, for timing one build
against another: which calls, on which sizes and inputs, and what the same
calculation gives in plain 64-bit torch.

A case is a dict of plain values; `prepare` makes what a program has in hand
before the call (seeded inputs on the device, plans, buffers), `run` is one
pass through the public entry points, `work` the bytes and operations a pass
cannot do without, `exact` the pass's result by ordinary torch arithmetic in
double precision.

Steps of an evolution start from a kept copy of the state (the copy a driver
keeps to be able to repeat a rejected step), so that every pass does the same
work on the same values.
"""
import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_1307_6488_gb300 import binding as B
from paper_1307_6488_gb300 import inputs

DEV = "cuda" if torch.cuda.is_available() else "cpu"
F64 = torch.float64
NV = 24
W, GT, TRK, AT, GAM, AL, BE, BB = 0, 1, 7, 8, 14, 17, 18, 21
SYM = ((0, 1, 2), (1, 3, 4), (2, 4, 5))
PAIRS = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))
CH = 32  # channels of the corrector network (24 used at its ends)
LAYER = 27 * CH * CH + CH
CFD_ITERATIONS = 4


# ------------------------------------------------------------------ the cases
def listed():
    bl = dict(data="bl", order=8, ghost=5)
    return [
        # the smallest grid in use: the gauge-wave stability test, periodic, where launches and latency count
        dict(name="rk4_fp64_24", op="rk4", prec="fp64", data="gauge_wave", order=4, ghost=3, nx=24, ny=24, nz=24),
        # the headline: a binary black hole grid, 8th order, static outer boundary
        dict(name="rk4_fp64_128", op="rk4", prec="fp64", nx=128, ny=128, nz=128, **bl),
        # the paper's integrator on a ragged grid near its single-GPU benchmark size (100^3)
        dict(name="rk3_fp64_odd", op="rk3", prec="fp64", nx=101, ny=93, nz=87, **bl),
        # the large production grid with a single-precision right-hand side
        dict(name="rk4_fp32_256", op="rk4", prec="fp32", nx=256, ny=256, nz=256, **bl),
        # the coarse step of a half-resolution run, 4th order, odd sizes
        dict(name="rk4_fp32_odd", op="rk4", prec="fp32", data="bl", order=4, ghost=4, nx=67, ny=61, nz=53),
        # uneven refinement patches around two punctures in one plan, both precisions
        dict(name="batch_fp64", op="batch", prec="fp64", order=4, ghost=4, blocks=32, tree=6488),
        dict(name="batch_fp32", op="batch", prec="fp32", order=4, ghost=4, blocks=96, tree=6488),
        # one coarse step of a refined hierarchy with subcycling (4 levels, 26 patches)
        dict(name="amr_fp64", op="amr", prec="fp64", order=8, ghost=5, n0=48, nested=3, fine_half=8, split=2),
        # the constraint monitor of an evolution, fields and norms
        dict(name="constraints_128", op="constraints", nx=128, ny=128, nz=128, **bl),
        # the learned corrector serving one step, and one training step on a batch
        dict(name="corrector_infer_64", op="infer", n=64, samples=1),
        dict(name="corrector_train_64", op="train", n=64, samples=4),
        # the second workload: lid-driven cavity of the CFD benchmark at its published size
        dict(name="cfd_256", op="cfd", nx=256, ny=256, nz=256, px=0, py=0, pz=0, alpha=0.3),
    ]


def draw(rng):
    """One more case from the ranges that the listed ones stand for."""
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def box(lo, hi):  # three axes around one size, so that the cost stays in range
        n = size(lo, hi)
        return {a: max(lo, min(hi, int(round(n * rng.uniform(0.75, 1.3))))) for a in ("nx", "ny", "nz")}

    op = rng.choice(["rk4", "rk4", "rk3", "rk4_32", "rk4_32", "batch", "amr", "constraints", "corrector", "cfd"])
    order = rng.choice([4, 8])
    ghost = order // 2 + 1 + rng.choice([0, 0, 1])
    if op in ("rk4", "rk3"):
        data = rng.choice(["bl", "gauge_wave"])
        return dict(op=op, prec="fp64", data=data, order=order, ghost=ghost, **box(12, 124))
    if op == "rk4_32":
        return dict(op="rk4", prec="fp32", data="bl", order=order, ghost=ghost, **box(16, 240))
    if op == "batch":
        return dict(op="batch", prec=rng.choice(["fp64", "fp32"]), order=order, ghost=ghost, blocks=size(2, 24),
                    tree=rng.randrange(1, 10000))
    if op == "amr":
        return dict(op="amr", prec=rng.choice(["fp64", "fp32"]), order=order, ghost=ghost,
                    n0=4 * rng.randrange(8, 13), nested=rng.choice([1, 2, 3]), fine_half=rng.choice([6, 7, 8]),
                    split=rng.choice([1, 2]))
    if op == "constraints":
        return dict(op=op, data=rng.choice(["bl", "gauge_wave"]), order=order, ghost=ghost, **box(12, 124))
    if op == "corrector":
        n = rng.choice([32, 64, 128])
        if n == 64 and rng.random() < 0.6:
            return dict(op="train", n=64, samples=rng.choice([1, 2, 3]))
        return dict(op="infer", n=n, samples=rng.choice([2, 3, 4]) if n < 128 else 1)
    per = {k: rng.choice([0, 0, 1]) for k in ("px", "py", "pz")}
    n = {k: 2 * (v // 2) if per["p" + k[1]] else v for k, v in box(16, 240).items()}
    return dict(op="cfd", alpha=round(rng.uniform(0.0, 1.0), 2), **n, **per)


# ------------------------------------------------------------------ inputs
def _params(case):
    return B.make_params(fd_order=case["order"], ko_eps=0.1, lapse=0, shift=0, eta=2.0)


def _prec(case):
    return B.FP32_RHS if case.get("prec") == "fp32" else B.FP64


def _waves(rs, extent):
    """Per variable three plane waves: wave vectors (one to three cycles over the extent), phases, amplitudes."""
    k = rs.uniform(-3.0, 3.0, (NV, 3, 3)) * (2 * np.pi / extent)
    return k, rs.uniform(0, 2 * np.pi, (NV, 3)), rs.uniform(0.2, 1.0, (NV, 3))


def _add_waves(u, x, y, z, waves, amplitude):
    k, phase, a = waves
    for v in range(NV):
        for w in range(3):
            u[v] += (amplitude * a[v, w]) * torch.sin(k[v, w, 0] * x + (k[v, w, 1] * y + (k[v, w, 2] * z + phase[v, w])))
    return u


def _axes(origin, n, g, h):
    """Cell centres of the padded points of a box, shaped to broadcast over (z, y, x)."""
    c = [origin[a] + (torch.arange(-g, n[a] + g, dtype=F64, device=DEV) + 0.5) * h for a in range(3)]
    return c[0][None, None, :], c[1][None, :, None], c[2][:, None, None]


def _bl_box(origin, n, g, h, holes, waves, amplitude=1e-3):
    """Two punctures (W = alpha = psi^-2) with every variable in motion: a small smooth wave field on top."""
    x, y, z = _axes(origin, n, g, h)
    psi = torch.ones((n[2] + 2 * g, n[1] + 2 * g, n[0] + 2 * g), dtype=F64, device=DEV)
    for m, c in holes:
        psi += m / (2 * torch.sqrt((x - c[0]) ** 2 + (y - c[1]) ** 2 + (z - c[2]) ** 2))
    u = torch.zeros((NV, *psi.shape), dtype=F64, device=DEV)
    u[W] = psi ** -2
    u[AL] = u[W]
    for i in range(3):
        u[GT + SYM[i][i]] = 1.0
    return _add_waves(u, x, y, z, waves, amplitude)


def _holes(rs):
    """Seeded masses and places near the x axis; 0.03 keeps them off the cell centres in use."""
    return [(rs.uniform(0.3, 0.7), (s * rs.uniform(1.3, 1.6), 0.03 * rs.uniform(0.5, 1), 0.03 * rs.uniform(0.5, 1)))
            for s in (-1, 1)]


def _wrap(u, g):
    for axis in (1, 2, 3):
        n = u.shape[axis] - 2 * g
        u = u.index_select(axis, torch.arange(-g, n + g, device=u.device) % n + g)
    return u


def _gauge_wave(case, rs, seed):
    """Gauge wave along x on [-1/2, 1/2] with the seeded 1e-10 noise of the stability test, periodic."""
    n, g = (case["nx"], case["ny"], case["nz"]), case["ghost"]
    h = 1.0 / n[0]
    x = _axes((-0.5,) * 3, n, 0, h)[0]
    A, ph = rs.uniform(0.008, 0.05), rs.uniform(0, 2 * np.pi)
    s, c = torch.sin(2 * np.pi * x + ph), torch.cos(2 * np.pi * x + ph)
    H, dH, K = 1 - A * s, -2 * np.pi * A * c, -np.pi * A * c / torch.sqrt(1 - A * s)
    u = torch.zeros((NV, n[2], n[1], n[0]), dtype=F64, device=DEV)
    u[W], u[AL] = H ** (-1 / 6), torch.sqrt(H)
    u[GT], u[GT + 3], u[GT + 5] = H ** (2 / 3), H ** (-1 / 3), H ** (-1 / 3)
    u[TRK], u[AT] = K / H, (2 / 3) * H ** (-1 / 3) * K
    u[AT + 3] = u[AT + 5] = -(1 / 3) * H ** (-4 / 3) * K
    u[GAM] = (2 / 3) * H ** (-5 / 3) * dH
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    u += 1e-10 * (2 * torch.rand(u.shape, dtype=F64, device=DEV, generator=gen) - 1)
    pad = torch.zeros((NV, n[2] + 2 * g, n[1] + 2 * g, n[0] + 2 * g), dtype=F64, device=DEV)
    pad[:, g:-g, g:-g, g:-g] = u
    return _wrap(pad, g), h


def _single(case, seed):
    """Initial data of a single grid: (state, spacing, boundary: 0 periodic, 1 static)."""
    rs = np.random.RandomState(seed % (1 << 32))
    if case["data"] == "gauge_wave":
        return (*_gauge_wave(case, rs, seed), 0)
    n = (case["nx"], case["ny"], case["nz"])
    h = 16.0 / max(n)
    waves, holes = _waves(rs, 16.0), _holes(rs)
    return _bl_box([-0.5 * m * h for m in n], n, case["ghost"], h, holes, waves), h, 1


def _blocks(case, seed):
    """Seeded refinement patches around two punctures: list of (state, n, h) and the common step."""
    rs = np.random.RandomState(seed % (1 << 32))
    holes, waves = _holes(rs), _waves(rs, 8.0)
    tree = inputs.patch_tree(nblocks=case["blocks"], seed=case["tree"], sides=tuple(range(16, 65, 6)))
    out = [(_bl_box(b["origin"], b["n"], case["ghost"], b["h"], holes, waves), b["n"], b["h"]) for b in tree]
    return out, 0.25 * min(b["h"] for b in tree)


def _amr_geometry(case):
    ncells, xlo, h0, geo = inputs.bl_hierarchy(n0=case["n0"], nested=case["nested"], fine_half=case["fine_half"],
                                               split=case["split"], extent=6.0 * 2 ** case["nested"])
    return ncells, xlo, h0, geo


def _amr_boxes(case, seed):
    """State of a box of cells of one level (padded), as a function (level, origin, n)."""
    rs = np.random.RandomState(seed % (1 << 32))
    _, xlo, h0, _ = _amr_geometry(case)
    holes, waves = _holes(rs), _waves(rs, -2 * xlo[0])

    def box(level, o, n):
        h = h0 / 2 ** level
        return _bl_box([xlo[a] + o[a] * h for a in range(3)], n, case["ghost"], h, holes, waves, amplitude=3e-4)
    return box


def _network(case, seed):
    """Seeded weights in the packed layout and BF16 inputs of the size normalised data has."""
    rs = np.random.RandomState(seed % (1 << 32))
    ch = [24, 32, 32, 32, 32, 24]
    p = np.zeros((5, LAYER), dtype=np.float32)
    for l in range(5):
        w = np.zeros((27, CH, CH))
        w[:, :ch[l + 1], :ch[l]] = rs.uniform(-1, 1, (27, ch[l + 1], ch[l])) * math.sqrt(6.0 / (27 * ch[l]))
        b = np.zeros(CH)
        b[:ch[l + 1]] = rs.uniform(-0.1, 0.1, ch[l + 1])
        p[l] = np.concatenate([w.ravel(), b])
    gen = torch.Generator(device=DEV).manual_seed(int(seed) + 1)
    shape = (case["samples"], case["n"], case["n"], case["n"], CH)
    x = torch.randn(shape, device=DEV, generator=gen)
    t = torch.randn(shape, device=DEV, generator=gen)
    x[..., 24:] = 0
    t[..., 24:] = 0
    return p.ravel(), x.to(torch.bfloat16), t.to(torch.bfloat16)


def _cfd_desc(case):
    n = (case["nx"], case["ny"], case["nz"])
    per = (case["px"], case["py"], case["pz"])
    h = 1.0 / max(n)
    return B.make_cfd(n, h, per, nu=1e-3, dt=0.25 * h, omega=1.7, alpha=case["alpha"], lid=1.0), n, h, per


def _flow(case, seed):
    """Smooth seeded velocities and pressure (ghost layers are set by the step itself)."""
    rs = np.random.RandomState(seed % (1 << 32))
    _, n, h, _ = _cfd_desc(case)
    x, y, z = _axes((0.0,) * 3, n, 1, h)
    out = []
    for c in range(4):
        f = torch.zeros((n[2] + 2, n[1] + 2, n[0] + 2), dtype=F64, device=DEV)
        for w in range(3):
            k = 2 * np.pi * rs.randint(-2, 3, 3)
            f += 0.1 * rs.uniform(0.2, 1) * torch.sin(k[0] * x + k[1] * y + k[2] * z + rs.uniform(0, 2 * np.pi))
        out.append(f.to(torch.float32))
    return out


# ------------------------------------------------------------------ prepare and run
class _Handle:
    """A library handle, given back with the state that holds it."""

    def __init__(self, value, destroy):
        self.value, self._destroy = value, destroy

    def __del__(self):
        self._destroy(self.value)


def _upload(u, grid, out=None):
    out = B.alloc_state(grid) if out is None else out
    B.view4(out, grid).copy_(u)
    return out


def _interior(flat, grid, nvar=NV):
    g = grid.ghost
    return B.view4(flat, grid, nvar)[:, g:g + grid.nz, g:g + grid.ny, g:g + grid.nx]


def _pool(grids):
    """One allocation that holds a state of every grid, and the states in it."""
    whole = torch.zeros(NV * sum(gr.var_stride for gr in grids), dtype=F64, device=DEV)
    parts, at = [], 0
    for gr in grids:
        parts.append(whole[at:at + NV * gr.var_stride])
        at += NV * gr.var_stride
    return whole, parts


def prepare(case, seed):
    op = case["op"]
    s = SimpleNamespace(case=case, op=op)
    if op in ("rk4", "rk3", "constraints"):
        u, h, s.bc = _single(case, seed)
        s.grid = B.make_grid(case["nx"], case["ny"], case["nz"], ghost=case["ghost"], dx=h)
        s.params, s.prec, s.dt = _params(case), _prec(case), 0.25 * h
        s.first = _upload(u, s.grid)
        s.work = B.alloc_work(s.grid, s.params, s.prec)
        if op == "constraints":
            s.ham = torch.zeros(s.grid.var_stride, dtype=F64, device=DEV)
            s.mom = torch.zeros(3 * s.grid.var_stride, dtype=F64, device=DEV)
            s.gcon = torch.zeros(3 * s.grid.var_stride, dtype=F64, device=DEV)
        else:
            s.state = s.first.clone()
            s.bufs = B.alloc_state(s.grid, n=3 if op == "rk4" else 2)
    elif op == "batch":
        blocks, s.dt = _blocks(case, seed)
        s.grids = [B.make_grid(*n, ghost=case["ghost"], dx=h) for _, n, h in blocks]
        s.first, src = _pool(s.grids)
        for (u, _, _), gr, part in zip(blocks, s.grids, src):
            _upload(u, gr, part)
        s.whole = s.first.clone()
        s.states, at = [], 0
        for gr in s.grids:
            s.states.append(s.whole[at:at + NV * gr.var_stride])
            at += NV * gr.var_stride
        s.plan = _Handle(B.plan_create(list(zip(s.grids, s.states, src)), _params(case), _prec(case)), B.plan_destroy)
    elif op == "amr":
        ncells, xlo, h0, geo = _amr_geometry(case)
        box = _amr_boxes(case, seed)
        s.grids = [B.make_grid(*n, ghost=case["ghost"], dx=h0 / 2 ** lev) for lev, _, n in geo]
        s.first, src = _pool(s.grids)
        for (lev, o, n), gr, part in zip(geo, s.grids, src):
            _upload(box(lev, o, n), gr, part)
        s.whole = s.first.clone()
        s.states, at = [], 0
        for gr in s.grids:
            s.states.append(s.whole[at:at + NV * gr.var_stride])
            at += NV * gr.var_stride
        patches = [(lev, o, n, gr.var_stride, st, f if lev == 0 else None)
                   for (lev, o, n), gr, st, f in zip(geo, s.grids, s.states, src)]
        s.amr = _Handle(B.amr_create(patches, ncells, xlo, h0, case["ghost"], 1, 0.25 * h0, _params(case),
                                     _prec(case)), B.amr_destroy)
    elif op in ("infer", "train"):
        p, s.x, s.t = _network(case, seed)
        s.net = _Handle(B.corrector_create(case["n"], case["samples"], seed=1), B.corrector_destroy)
        B.corrector_params(s.net.value, p)
        s.out = torch.empty((case["samples"], case["n"] ** 3, CH), dtype=torch.float32, device=DEV)
    else:
        s.desc = _cfd_desc(case)[0]
        s.fields = _flow(case, seed)
        s.scratch = torch.empty(3 * ((B.cfd_points(s.desc) + 3) // 4 * 4), dtype=torch.float32, device=DEV)
    return s


def run(s):
    op = s.op
    if op == "rk4":
        s.state.copy_(s.first)
        B.rk4_step(s.grid, s.params, s.prec, s.dt, s.bc, s.first if s.bc else None, s.state, s.bufs, s.work)
        return _interior(s.state, s.grid)
    if op == "rk3":
        s.state.copy_(s.first)
        B.rk3_step(s.grid, s.params, s.prec, s.dt, s.bc, s.first if s.bc else None, s.state, s.bufs, s.work)
        return _interior(s.state, s.grid)
    if op == "constraints":
        l2, mx, _ = B.constraints(s.grid, s.params, s.first, s.work, s.ham, s.mom, s.gcon)
        return [_interior(s.ham, s.grid, 1), _interior(s.mom, s.grid, 3), _interior(s.gcon, s.grid, 3), l2, mx]
    if op == "batch":
        s.whole.copy_(s.first)
        B.batch_step(s.plan.value, s.dt)
        return s.whole  # every patch, ghosts included, in the order of the plan
    if op == "amr":
        s.whole.copy_(s.first)
        B.amr_step(s.amr.value)
        return [_interior(st, gr) for st, gr in zip(s.states, s.grids)]
    if op == "infer":
        B.corrector_infer_async(s.net.value, s.case["samples"], s.x, s.out)
        return s.out
    if op == "train":
        loss = B.corrector_train_step_raw(s.net.value, list(s.x), list(s.t), 1e-4)
        return [loss, B.corrector_grads(s.net.value).reshape(5, LAYER)]
    B.cfd_step(s.desc, CFD_ITERATIONS, *s.fields, s.scratch)
    return list(s.fields)


# ------------------------------------------------------------------ work
def _step_flops(order):
    """Operations of one point and Runge-Kutta stage: stencils, algebra, dissipation, update."""
    H, r = order // 2, order // 2 + 1
    stencils = 45 * 3 * H + 33 * (5 * H + 1) + 33 * 3 * H + 72 * (4 * (order + 1) + 7) + 48
    return stencils + 3285 + 24 * (12 * r + 10) + 96


def _padded(n, g):
    return (n[0] + 2 * g) * (n[1] + 2 * g) * (n[2] + 2 * g)


def work(case):
    op = case["op"]
    if op in ("rk4", "rk3", "constraints"):
        n = (case["nx"], case["ny"], case["nz"])
        pts, pad = math.prod(n), _padded(n, case["ghost"])
        if op == "constraints":
            H = case["order"] // 2
            per_point = 51 * 3 * H + 21 * (5 * H + 1) + 21 * 3 * H + 2000
            return {"bytes": 8 * NV * pad + 8 * 7 * pts, "flops": per_point * pts}
        stages = 4 if op == "rk4" else 3
        return {"bytes": 8 * NV * (pad + pts), "flops": stages * _step_flops(case["order"]) * pts}
    if op == "batch":
        tree = inputs.patch_tree(nblocks=case["blocks"], seed=case["tree"], sides=tuple(range(16, 65, 6)))
        pts = sum(math.prod(b["n"]) for b in tree)
        pad = sum(_padded(b["n"], case["ghost"]) for b in tree)
        return {"bytes": 8 * NV * (pad + pts), "flops": 4 * _step_flops(case["order"]) * pts}
    if op == "amr":
        geo = _amr_geometry(case)[3]
        updates = sum(math.prod(n) * 2 ** lev for lev, _, n in geo)
        size = sum(math.prod(n) + _padded(n, case["ghost"]) for _, _, n in geo)
        return {"bytes": 8 * NV * size, "flops": 4 * _step_flops(case["order"]) * updates}
    if op in ("infer", "train"):
        pts = case["samples"] * case["n"] ** 3
        flops = 2 * 27 * (24 * 32 + 3 * 32 * 32 + 32 * 24) * pts
        if op == "infer":
            return {"bytes": pts * CH * (2 + 4) + 4 * 5 * LAYER, "flops": flops}
        return {"bytes": pts * CH * (2 + 2) + 7 * 4 * 5 * LAYER, "flops": 3 * flops}
    cells = case["nx"] * case["ny"] * case["nz"]
    return {"bytes": 32 * cells, "flops": (207 + 22 * CFD_ITERATIONS) * cells}


# ------------------------------------------------------------------ the same in plain 64-bit torch
FD = {4: dict(d1=[2 / 3, -1 / 12], d2=[4 / 3, -1 / 12], lo=-1, up=[-3 / 12, -10 / 12, 18 / 12, -6 / 12, 1 / 12],
              ko=[15.0, -6.0, 1.0], scale=1 / 64),
      8: dict(d1=[4 / 5, -1 / 5, 4 / 105, -1 / 280], d2=[8 / 5, -1 / 5, 8 / 315, -1 / 560], lo=-3,
              up=[-1 / 168, 1 / 14, -1 / 2, -9 / 20, 5 / 4, -1 / 2, 1 / 6, -1 / 28, 1 / 280],
              ko=[210.0, -120.0, 45.0, -10.0, 1.0], scale=1 / 1024)}
KO_EPS, ETA, SHIFT = 0.1, 2.0, 0.75


class _Stencils:
    """Derivatives at the interior points of one padded variable, axis 0 = x."""

    def __init__(self, g, h, order):
        self.g, self.h, self.f = g, h, FD[order]

    def at(self, v, off, ext=(0, 0, 0)):
        """v shifted by off = (x, y, z), on the interior widened by ext points."""
        return v[tuple(slice(self.g - ext[a] + off[a], v.shape[2 - a] - self.g + ext[a] + off[a]) for a in (2, 1, 0))]

    @staticmethod
    def _e(a, o):
        return tuple(o if b == a else 0 for b in range(3))

    def d1(self, v, a, ext=(0, 0, 0)):
        return sum(c * (self.at(v, self._e(a, o + 1), ext) - self.at(v, self._e(a, -o - 1), ext))
                   for o, c in enumerate(self.f["d1"])) / self.h

    def d2(self, v, a, b):
        if a == b:
            c0 = 2 * self.at(v, (0, 0, 0))
            return sum(c * ((self.at(v, self._e(a, o + 1)) + self.at(v, self._e(a, -o - 1))) - c0)
                       for o, c in enumerate(self.f["d2"])) / self.h ** 2
        out = 0
        H = len(self.f["d1"])
        first = self.d1(v, a, self._e(b, H))  # widened along b
        ax = 2 - b
        m = first.shape[ax] - 2 * H
        for o, c in enumerate(self.f["d1"]):
            out = out + c * (first.narrow(ax, H + o + 1, m) - first.narrow(ax, H - o - 1, m))
        return out / self.h

    def advect(self, v, beta):
        out = 0
        for a in range(3):
            fwd = sum(c * self.at(v, self._e(a, self.f["lo"] + i)) for i, c in enumerate(self.f["up"]))
            bwd = sum(c * self.at(v, self._e(a, -self.f["lo"] - i)) for i, c in enumerate(self.f["up"]))
            out = out + torch.where(beta[a] >= 0, beta[a] * fwd, -beta[a] * bwd)
        return out / self.h

    def dissipate(self, v):
        c0 = 2 * self.at(v, (0, 0, 0))
        out = sum(c * ((self.at(v, self._e(a, o + 1)) + self.at(v, self._e(a, -o - 1))) - c0)
                  for a in range(3) for o, c in enumerate(self.f["ko"]))
        return out * (KO_EPS * self.f["scale"] / self.h)


R3 = range(3)


def _geometry(S, u):
    """Inverse metric, Christoffel symbols and Ricci tensor of the BSSN variables at the interior points."""
    c = [S.at(u[v], (0, 0, 0)) for v in range(NV)]
    g = [[c[GT + SYM[i][j]] for j in R3] for i in R3]
    cof = [[g[(i + 1) % 3][(j + 1) % 3] * g[(i + 2) % 3][(j + 2) % 3]
            - g[(i + 1) % 3][(j + 2) % 3] * g[(i + 2) % 3][(j + 1) % 3] for j in R3] for i in R3]
    det = sum(g[0][j] * cof[0][j] for j in R3)
    gu = [[cof[i][j] / det for j in R3] for i in R3]
    dg = [[[None] * 3 for _ in R3] for _ in R3]  # dg[k][i][j] = d_k g_ij
    for k in R3:
        for i, j in PAIRS:
            dg[k][i][j] = dg[k][j][i] = S.d1(u[GT + SYM[i][j]], k)
    low = [[[0.5 * (dg[i][k][j] + dg[j][k][i] - dg[k][i][j]) for j in R3] for i in R3] for k in R3]
    up = [[[sum(gu[k][l] * low[l][i][j] for l in R3) for j in R3] for i in R3] for k in R3]
    gd = [sum(gu[i][j] * up[k][i][j] for i in R3 for j in R3) for k in R3]
    dgam = [[S.d1(u[GAM + i], d) for i in R3] for d in R3]
    dW = [S.d1(u[W], d) for d in R3]
    iw = 1 / c[W]
    ddw = [[None] * 3 for _ in R3]
    for i, j in PAIRS:
        ddw[i][j] = ddw[j][i] = S.d2(u[W], i, j) - sum(up[k][i][j] * dW[k] for k in R3)
    tr = sum(gu[i][j] * ddw[i][j] for i in R3 for j in R3)
    dwdw = sum(gu[i][j] * dW[i] * dW[j] for i in R3 for j in R3)
    ric = [[None] * 3 for _ in R3]
    mixed = [[[sum(gu[l][m] * low[j][k][m] for m in R3) for l in R3] for k in R3] for j in R3]  # G_jk^l
    for i, j in PAIRS:
        v = u[GT + SYM[i][j]]
        r = -0.5 * sum((1 if a == b else 2) * gu[a][b] * S.d2(v, a, b) for a, b in PAIRS)
        r = r + 0.5 * sum(g[k][i] * dgam[j][k] + g[k][j] * dgam[i][k] + gd[k] * (low[i][j][k] + low[j][i][k])
                          for k in R3)
        r = r + sum(up[k][l][i] * mixed[j][k][l] + up[k][l][j] * mixed[i][k][l] + up[k][i][l] * mixed[k][j][l]
                    for k in R3 for l in R3)
        r = r + ddw[i][j] * iw + g[i][j] * (tr - 2 * dwdw * iw) * iw
        ric[i][j] = ric[j][i] = r
    return SimpleNamespace(c=c, g=g, gu=gu, up=up, gd=gd, dW=dW, iw=iw, ric=ric)


def _rhs(u, g, h, order):
    """Right-hand side (1+log, Gamma-driver, advected gauge) with dissipation, interior points."""
    S = _Stencils(g, h, order)
    G = _geometry(S, u)
    c, gt, gu, up = G.c, G.g, G.gu, G.up
    A = [[c[AT + SYM[i][j]] for j in R3] for i in R3]
    K, al, beta = c[TRK], c[AL], [c[BE + i] for i in R3]
    Am = [[sum(gu[i][k] * A[k][j] for k in R3) for j in R3] for i in R3]
    Au = [[sum(Am[i][k] * gu[k][j] for k in R3) for j in R3] for i in R3]
    AA = sum(A[i][j] * Au[i][j] for i in R3 for j in R3)
    da = [S.d1(u[AL], d) for d in R3]
    dWda = sum(gu[i][j] * G.dW[i] * da[j] for i in R3 for j in R3)
    dda, X = [[None] * 3 for _ in R3], [[None] * 3 for _ in R3]
    for i, j in PAIRS:
        dda[i][j] = dda[j][i] = (S.d2(u[AL], i, j) - sum(up[k][i][j] * da[k] for k in R3)
                                 + (G.dW[i] * da[j] + G.dW[j] * da[i] - gt[i][j] * dWda) * G.iw)
        X[i][j] = X[j][i] = al * G.ric[i][j] - dda[i][j]
    trX = sum(gu[i][j] * X[i][j] for i in R3 for j in R3)
    db = [[S.d1(u[BE + i], d) for i in R3] for d in R3]  # db[d][i]
    div = db[0][0] + db[1][1] + db[2][2]
    out = [None] * NV
    out[W] = c[W] / 3 * (al * K - div)
    out[TRK] = -c[W] ** 2 * sum(gu[i][j] * dda[i][j] for i in R3 for j in R3) + al * (AA + K * K / 3)
    for i, j in PAIRS:
        s = SYM[i][j]
        out[GT + s] = (-2 * al * A[i][j] + sum(gt[i][k] * db[j][k] + gt[j][k] * db[i][k] for k in R3)
                       - 2 / 3 * div * gt[i][j])
        out[AT + s] = (c[W] ** 2 * (X[i][j] - trX * gt[i][j] / 3)
                       + al * (K * A[i][j] - 2 * sum(A[i][k] * Am[k][j] for k in R3))
                       + sum(A[i][k] * db[j][k] + A[j][k] * db[i][k] for k in R3) - 2 / 3 * div * A[i][j])
    dK = [S.d1(u[TRK], d) for d in R3]
    dd = [[[None] * 3 for _ in R3] for _ in R3]
    for i in R3:
        for j, k in PAIRS:
            dd[i][j][k] = dd[i][k][j] = S.d2(u[BE + i], j, k)
    for i in R3:
        r = sum(gu[j][k] * dd[i][j][k] for j in R3 for k in R3)
        r = r + sum(gu[i][j] * dd[k][j][k] for j in R3 for k in R3) / 3
        r = r - sum(G.gd[j] * db[j][i] for j in R3) + 2 / 3 * div * G.gd[i]
        r = r - 2 * sum(Au[i][j] * da[j] for j in R3)
        r = r + 2 * al * (sum(up[i][j][k] * Au[j][k] for j in R3 for k in R3)
                          - 3 * G.iw * sum(Au[i][j] * G.dW[j] for j in R3)
                          - 2 / 3 * sum(gu[i][j] * dK[j] for j in R3))
        out[GAM + i] = r
        out[BB + i] = r - ETA * c[BB + i]
        out[BE + i] = SHIFT * c[BB + i]
    out[AL] = -2 * al * K
    for v in range(NV):
        out[v] = out[v] + S.advect(u[v], beta) + S.dissipate(u[v])
    return torch.stack(out)


def _rk_step(u, g, h, order, dt, ghosts, method="rk4", keep=False):
    """One step; ghosts(x, s) sets the ghost points of the input of stage s (and of the result, s = 4)."""
    inn = (slice(None), slice(g, -g), slice(g, -g), slice(g, -g))

    def with_interior(x, s):
        y = u.clone()
        y[inn] = x
        return ghosts(y, s)

    y0 = u[inn].clone()
    if method == "rk3":
        y = y0 + dt * _rhs(u, g, h, order)
        y = 0.75 * y0 + 0.25 * (y + dt * _rhs(with_interior(y, 1), g, h, order))
        y = y0 / 3 + 2 / 3 * (y + dt * _rhs(with_interior(y, 2), g, h, order))
        return with_interior(y, 4)
    stages = [u]
    total = 0
    for s, (b, a) in enumerate(((1, 0.5), (2, 0.5), (2, 1.0), (1, None))):
        k = _rhs(stages[-1], g, h, order)
        total = total + b / 6 * dt * k
        if a is not None:
            stages.append(with_interior(y0 + a * dt * k, s + 1))
    out = with_interior(y0 + total, 4)
    return (out, stages + [out]) if keep else out


def _static(first, g):
    def ghosts(x, s):
        y = first.clone()
        y[:, g:-g, g:-g, g:-g] = x[:, g:-g, g:-g, g:-g]
        return y
    return ghosts


# the refined hierarchy: every level below the finest is one box cut into patches, the finest two boxes apart
_PROLONG = ((-5 / 128, 35 / 128, 105 / 128, -7 / 128), (-7 / 128, 105 / 128, 35 / 128, -5 / 128))


def _prolong(f, fo, o, n, g):
    """Tricubic values of the parent field f (padded, first interior cell fo) at the padded cells of a fine box."""
    for a in range(3):
        cell = torch.arange(o[a] - g, o[a] + n[a] + g, device=f.device)
        odd = cell % 2
        base = torch.div(cell, 2, rounding_mode="floor") - 2 + odd - (fo[a] - g)
        wts = torch.tensor(_PROLONG, dtype=F64, device=f.device)[odd]
        shape = [1] * 4
        shape[3 - a] = -1
        f = sum(wts[:, j].reshape(shape) * f.index_select(3 - a, base + j) for j in range(4))
    return f


def _dense(half, stage):
    """Weights over (Y2, Y3, Y4, y1) - y0 of the parent's step that give the fine ghost at a stage input."""
    c1 = np.array([2.0, 0, 0, 0])
    k2, k3, k4 = np.array([0, 2.0, 0, 0]), np.array([0, 0, 1.0, 0]), np.array([-2.0, -4, -2, 6])
    c2, c3 = -1.5 * c1 + k2 + k3 - 0.5 * k4, 2 / 3 * (c1 - k2 - k3 + k4)
    x = 0.5 * half + (0.5 if stage == 4 else 0.0)
    y = x * c1 + x ** 2 * c2 + x ** 3 * c3
    d1, d2, d3 = c1 + 2 * x * c2 + 3 * x ** 2 * c3, 2 * c2 + 6 * x * c3, 6 * c3
    if stage in (0, 4):
        return y
    if stage == 1:
        return y + 0.25 * d1
    if stage == 2:
        return y + 0.25 * d1 + d2 / 16
    return y + 0.5 * d1 + d2 / 8 + d3 / 32


def _exact_amr(case, seed):
    ncells, xlo, h0, geo = _amr_geometry(case)
    g, make = case["ghost"], _amr_boxes(case, seed)
    boxes = []  # per level: [origin, n, state]
    for lev in range(case["nested"] + 1):
        mine = [(o, n) for l, o, n in geo if l == lev]
        if lev < case["nested"]:
            lo = tuple(min(o[a] for o, _ in mine) for a in range(3))
            mine = [(lo, tuple(max(o[a] + n[a] for o, n in mine) - lo[a] for a in range(3)))]
        boxes.append([[o, n, make(lev, o, n)] for o, n in mine])
    fixed = boxes[0][0][2].clone()

    def advance(lev, half, parent):
        for b in boxes[lev]:
            o, n, _ = b
            if lev == 0:
                ghosts = _static(fixed, g)
            else:
                pre = [_prolong(f, boxes[lev - 1][0][0], o, n, g) for f in parent]

                def ghosts(x, s, pre=pre):
                    y = pre[0] + sum(float(w) * p for w, p in zip(_dense(half, s), pre[1:]))
                    y[:, g:-g, g:-g, g:-g] = x[:, g:-g, g:-g, g:-g]
                    return y
            b[2], stages = _rk_step(ghosts(b[2], 0), g, h0 / 2 ** lev, case["order"], 0.25 * h0 / 2 ** lev, ghosts,
                                    keep=True)
        if lev == case["nested"]:
            return
        fields = [stages[0]] + [x - stages[0] for x in stages[1:]]
        for k in (0, 1):
            advance(lev + 1, k, fields)
        co, _, cs = boxes[lev][0]
        for l, po, pn in geo:  # each finer patch covers the coarse cells whose 4-cell runs lie inside it
            if l != lev + 1:
                continue
            fo, _, fine = next(b for b in boxes[l] if all(b[0][a] <= po[a] < b[0][a] + b[1][a] for a in R3))
            f, dst = fine, [slice(None)]
            for a in R3:
                c = torch.arange((po[a] + 2) // 2, (po[a] + pn[a] - 3) // 2 + 1, device=f.device)
                base = 2 * c - 1 - fo[a] + g
                f = sum(w / 16 * f.index_select(3 - a, base + j) for j, w in enumerate((-1.0, 9.0, 9.0, -1.0)))
                dst.insert(1, slice(int(c[0]) - co[a] + g, int(c[-1]) + 1 - co[a] + g))
            cs[tuple(dst)] = f

    advance(0, 0, None)
    out = []
    for lev, o, n in geo:
        bo, _, st = next(b for b in boxes[lev] if all(b[0][a] <= o[a] < b[0][a] + b[1][a] for a in R3))
        at = [o[a] - bo[a] + g for a in R3]
        out.append(st[:, at[2]:at[2] + n[2], at[1]:at[1] + n[1], at[0]:at[0] + n[0]])
    return out


def _exact_constraints(u, g, h, order):
    S = _Stencils(g, h, order)
    G = _geometry(S, u)
    c, gu, up = G.c, G.gu, G.up
    A = [[c[AT + SYM[i][j]] for j in R3] for i in R3]
    Am = [[sum(gu[i][k] * A[k][j] for k in R3) for j in R3] for i in R3]
    scal = c[W] ** 2 * sum(gu[i][j] * G.ric[i][j] for i in R3 for j in R3)
    ham = scal + 2 / 3 * c[TRK] ** 2 - sum(Am[i][j] * Am[j][i] for i in R3 for j in R3)
    dA = [[[None] * 3 for _ in R3] for _ in R3]
    for k in R3:
        for i, j in PAIRS:
            dA[k][i][j] = dA[k][j][i] = S.d1(u[AT + SYM[i][j]], k)
    mom = []
    for i in R3:
        m = sum(gu[j][k] * (dA[k][i][j] - sum(up[l][k][i] * A[l][j] + up[l][k][j] * A[i][l] for l in R3))
                for j in R3 for k in R3)
        mom.append(m - 3 * G.iw * sum(Am[j][i] * G.dW[j] for j in R3) - 2 / 3 * S.d1(u[TRK], i))
    gcon = [c[GAM + i] - G.gd[i] for i in R3]
    every = torch.stack([ham] + mom + gcon).reshape(7, -1)
    l2, mx = every.square().mean(1).sqrt(), every.abs().amax(1)
    return [ham[None], torch.stack(mom), torch.stack(gcon), l2.cpu().numpy(), mx.cpu().numpy()]


def _gelu(x):
    return 0.5 * x * (1 + torch.tanh(math.sqrt(2 / math.pi) * (x + 0.044715 * x ** 3)))


def _exact_network(case, seed):
    p, x, t = _network(case, seed)
    p = torch.from_numpy(p).to(DEV).to(F64).requires_grad_(case["op"] == "train")
    n = case["n"]
    chunk, loss, outs = 1, 0.0, []
    for s in range(0, case["samples"], chunk):
        a = x[s:s + chunk].to(F64).permute(0, 4, 1, 2, 3)
        for l in range(5):
            w = p[l * LAYER:(l + 1) * LAYER - CH].reshape(3, 3, 3, CH, CH).permute(3, 4, 0, 1, 2)
            a = torch.nn.functional.conv3d(a, w, p[(l + 1) * LAYER - CH:(l + 1) * LAYER], padding=1)
            a = _gelu(a) if l < 4 else a
        a = a.permute(0, 2, 3, 4, 1)
        if case["op"] == "infer":
            outs.append(a.detach().reshape(chunk, n ** 3, CH))
            continue
        d = (a - t[s:s + chunk].to(F64))[..., :24]
        part = d.square().sum() / (case["samples"] * n ** 3 * 24)
        part.backward()
        loss += float(part.detach())
    if case["op"] == "infer":
        return torch.cat(outs)
    return [loss, p.grad.reshape(5, LAYER).cpu().numpy()]


def _exact_cfd(case, seed):
    d, n, h, per = _cfd_desc(case)
    dt, nu, al, om = d.dt, d.nu, d.alpha, d.omega
    u, v, w, p = (f.to(F64) for f in _flow(case, seed))
    vel = [u, v, w]

    def plane(a, i):
        s = [slice(None)] * 3
        s[2 - a] = i
        return tuple(s)

    def boundary():
        for a in R3:
            last = n[a]
            for c, f in enumerate(vel + [p]):
                if per[a]:
                    f[plane(a, 0)] = f[plane(a, last)]
                    f[plane(a, last + 1)] = f[plane(a, 1)]
                elif c == a:
                    f[plane(a, 0)] = f[plane(a, last)] = f[plane(a, last + 1)] = 0
                elif c == 3:
                    f[plane(a, 0)] = f[plane(a, 1)]
                    f[plane(a, last + 1)] = f[plane(a, last)]
                else:
                    f[plane(a, 0)] = -f[plane(a, 1)]
                    f[plane(a, last + 1)] = 2 * (d.lid if a == 2 and c == 0 else 0.0) - f[plane(a, last)]

    def at(f, off, end):
        return f[tuple(slice(1 + off[a], end[a] + off[a]) for a in (2, 1, 0))]

    def e(a, s):
        return tuple(s if b == a else 0 for b in R3)

    boundary()
    new = []
    for c in R3:
        end = [n[a] if a == c and not per[a] else n[a] + 1 for a in R3]
        f = vel[c]
        x = at(f, (0, 0, 0), end)
        r = (at(p, (0, 0, 0), end) - at(p, e(c, 1), end)) / h + d.g[c]
        for b in R3:
            hi, lo = at(f, e(b, 1), end), at(f, e(b, -1), end)
            if b == c:
                th, tl = x + hi, lo + x
            else:
                both = tuple(i + j for i, j in zip(e(b, -1), e(c, 1)))
                th = at(vel[b], (0, 0, 0), end) + at(vel[b], e(c, 1), end)
                tl = at(vel[b], e(b, -1), end) + at(vel[b], both, end)
            r = r - (th * (x + hi) + al * th.abs() * (x - hi) - tl * (lo + x) - al * tl.abs() * (lo - x)) / (4 * h)
            r = r + nu * (hi - 2 * x + lo) / h ** 2
        new.append((tuple(slice(1, end[a]) for a in (2, 1, 0)), x + dt * r))
    for f, (where, val) in zip(vel, new):
        f[where] = val
    boundary()
    cell = [torch.arange(n[a], device=DEV).reshape([-1 if 2 - a == q else 1 for q in R3]) for a in R3]
    colour = (cell[0] + cell[1] + cell[2]) % 2
    low = [torch.ones_like(cell[a], dtype=F64) if per[a] else (cell[a] > 0).to(F64) for a in R3]
    high = [torch.ones_like(cell[a], dtype=F64) if per[a] else (cell[a] < n[a] - 1).to(F64) for a in R3]
    beta = om / (dt * sum((low[a] + high[a]) / h ** 2 for a in R3))
    inn = (slice(1, -1),) * 3
    for _ in range(CFD_ITERATIONS):
        for col in (0, 1):
            div = sum((vel[a][inn] - at(vel[a], e(a, -1), [m + 1 for m in n])) / h for a in R3)
            dp = torch.where(colour == col, -beta * div, torch.zeros((), dtype=F64, device=DEV))
            p[inn] += dp
            for a in R3:
                vel[a][inn] += dt / h * dp * high[a]
                lows = dt / h * dp * low[a]
                vel[a][inn] -= torch.roll(lows, -1, 2 - a)  # the low face of cell i + 1 is the high face of cell i
                if per[a]:
                    vel[a][plane(a, 0)] = vel[a][plane(a, n[a])]
        boundary()
    return [u, v, w, p]


def exact(case, seed):
    op = case["op"]
    if op in ("rk4", "rk3", "constraints"):
        u, h, bc = _single(case, seed)
        g = case["ghost"]
        if op == "constraints":
            return _exact_constraints(u, g, h, case["order"])
        ghosts = _static(u.clone(), g) if bc else (lambda x, s: _wrap(x, g))
        return _rk_step(u, g, h, case["order"], 0.25 * h, ghosts, op)[:, g:-g, g:-g, g:-g]
    if op == "batch":
        blocks, dt = _blocks(case, seed)
        g = case["ghost"]
        whole, parts = _pool([B.make_grid(*n, ghost=g, dx=h) for _, n, h in blocks])
        for (u, n, h), part in zip(blocks, parts):
            _upload(_rk_step(u, g, h, case["order"], dt, _static(u.clone(), g)), B.make_grid(*n, ghost=g, dx=h), part)
        return whole
    if op == "amr":
        return _exact_amr(case, seed)
    if op in ("infer", "train"):
        return _exact_network(case, seed)
    return _exact_cfd(case, seed)
