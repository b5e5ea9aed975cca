"""The work that a reservoir simulator has this library do, as measurable cases.

A Newton step of the simulator hands over new Jacobian values, rebuilds the preconditioner and runs a
preconditioned Krylov solve; the cases are that path's single calls (matrix-vector product, preconditioner
application, preconditioner rebuild), its whole solves (an inexact one of one GMRES(30) cycle, a tight
mixed-precision one, an ensemble of small systems), and the convolutions of the learned pressure stage, forward and
backward.  Grids run from 4,000 cells, where launches and latency count, to 8.4 million.

Jacobians follow the repository's synthetic recipe (two-point flux on unit cells, log-normal, layered or channelised
permeability, row-diagonally dominant 3x3 mobility blocks, a small accumulation term), drawn on the GPU.

``exact`` restates each path in plain torch, 64 bits: natural-order block ILU(0) by i+j+k planes, the geometric
V-cycle, the CPR stage orders, textbook GMRES, and convolutions as sums of shifted matrix products.
"""
from __future__ import annotations

import ctypes
import math
import random

import torch

import paper_1602_05901_gb300 as rsv

DEV = "cuda"
SLOTS = ((0, 0, -1), (0, -1, 0), (-1, 0, 0), (0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1))  # (di, dj, dk), ascending column
STAGES = {"bilu0": "F", "cpr": "PF", "cpr_fp": "FP", "cpr_fpf": "FPF", "cpr_ffpf": "FFPF"}
CYCLE = 30        # GMRES restart length, and the linear iterations of an inexact Newton step
TIGHT = 1e-12     # relative tolerance of the fully converged solves


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # matrix-vector product of the FP64 outer residual, on the 100x100x50 configuration
        dict(name="spmv_f64_mid", kind="spmv", nx=100, ny=100, nz=50, prec="fp64", perm="layered"),
        # matrix-vector product of the FP32 inner solve, on the largest configuration
        dict(name="spmv_f32_large", kind="spmv", nx=256, ny=256, nz=128, prec="mixed", perm="channelized"),
        # block ILU(0) inside the FP32 inner solve, 100x100x50
        dict(name="ilu_f32_mid", kind="apply", nx=100, ny=100, nz=50, prec="mixed", pc="bilu0", perm="layered"),
        # block ILU(0) of a plain FP64 solve on a ragged grid (no side a multiple of a tile)
        dict(name="ilu_f64_ragged", kind="apply", nx=75, ny=61, nz=37, prec="fp64", pc="bilu0", perm="lognormal"),
        # the headline's preconditioner application: CPR (pressure V-cycle, then block ILU(0)) in FP32, 8.4M cells
        dict(name="cpr_f32_large", kind="apply", nx=256, ny=256, nz=128, prec="mixed", pc="cpr", perm="channelized"),
        # what every Newton step pays before its solve: new values, rebuilt CPR, first application (learned-stage grid)
        dict(name="newton_cpr_f32", kind="newton", nx=128, ny=128, nz=64, prec="mixed", pc="cpr", perm="channelized"),
        # an inexact Newton step of a small model: one GMRES(30) cycle in FP64; latency and launches
        dict(name="cycle_f64_tiny", kind="cycle", nx=20, ny=20, nz=10, prec="fp64", pc="bilu0", perm="lognormal"),
        # the same of a large model with the FPF stage order, FP64
        dict(name="cycle_f64_cpr_fpf", kind="cycle", nx=128, ny=128, nz=64, prec="fp64", pc="cpr_fpf", perm="channelized"),
        # a whole mixed-precision solve, FP32 inner GMRES(30) + CPR under FP64 refinement, converged tightly
        dict(name="solve_mixed_mid", kind="solve", nx=100, ny=100, nz=50, prec="mixed", pc="cpr", perm="lognormal"),
        # an ensemble of uneven small models in one batched solve (BiCGSTAB + block ILU(0), mixed precision)
        dict(name="ensemble_mixed", kind="batch", count=24, sizes=3, prec="mixed", pc="bilu0"),
        # the learned pressure stage's widest volume: one 3x3x3 convolution layer, bias and ReLU
        dict(name="conv_fwd_level0", kind="conv", nx=128, ny=128, nz=64, ci=32, co=32, direction="forward"),
        # training that stage: input, weight and bias gradients of one layer at the next level
        dict(name="conv_bwd_level1", kind="conv", nx=64, ny=64, nz=32, ci=64, co=64, direction="backward"),
    ]


def draw(rng):
    kind = rng.choice(["spmv", "apply", "apply", "newton", "cycle", "solve", "batch", "conv"])
    if kind == "conv":
        level = rng.randrange(4)
        return dict(kind="conv", nx=8 * rng.randint(1, 16 >> level), ny=rng.randint(6, 128 >> level) if level < 3 else rng.randint(4, 16),
                    nz=rng.randint(4, max(4, 64 >> level)), ci=rng.choice([32, 64, 96]) << min(level, 2),
                    co=rng.choice([32, 64]) << min(level, 2), direction=rng.choice(["forward", "backward"]))
    if kind == "batch":
        return dict(kind="batch", count=rng.randint(4, 20), sizes=rng.randrange(4, 1 << 20), prec="mixed", pc="bilu0")
    most = {"spmv": 8e6, "apply": 8e6, "newton": 1e6, "cycle": 1e6, "solve": 2e5}[kind]
    nx, ny, nz = _draw_grid(rng, 1e5 if kind == "spmv" else 4e3, most)  # a smaller product takes less than its launch
    case = dict(kind=kind, nx=nx, ny=ny, nz=nz, prec=rng.choice(["fp64", "mixed"]),
                perm=rng.choice(["lognormal", "layered", "channelized"]))
    if kind == "cycle":
        case.update(prec="fp64", pc=rng.choice(["bilu0", "cpr", "cpr_fpf"]))
    elif kind == "solve":
        case.update(prec="mixed", pc=rng.choice(["bilu0", "cpr"]), perm="lognormal")
    elif kind != "spmv":
        case.update(pc=rng.choice(["bilu0", "cpr", "cpr_fpf"]))
    return case


def _draw_grid(rng, least, most):
    """A grid of log-uniformly many cells; sides of any parity, the vertical one the shortest as a rule."""
    cells = math.exp(rng.uniform(math.log(least), math.log(most)))
    a, b = rng.uniform(0.7, 1.5), rng.uniform(0.3, 0.9)  # ny / nx, nz / nx
    nx = max(6, round((cells / (a * b)) ** (1 / 3)))
    ny = max(6, round(a * nx))
    return nx, ny, max(4, int(cells / (nx * ny)))


def _ensemble(case):
    r = random.Random(case["sizes"])
    return [(r.randint(16, 96), r.randint(16, 96), r.randint(16, 48)) for _ in range(case["count"])]


# ------------------------------------------------------------------ inputs

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _permeability(nx, ny, nz, kind, g, seed):
    """ln k per cell, [nz, ny, nx]."""
    z = torch.randn(nz, ny, nx, device=DEV, dtype=torch.float64, generator=g)
    mean = math.log(100.0)
    if kind == "layered":
        return mean + 1.5 * torch.randn(nz, 1, 1, device=DEV, dtype=torch.float64, generator=g) + 0.5 * z
    if kind == "lognormal":
        return mean + z
    lnk = mean + 2.0 * z
    streaks = torch.zeros(nz, ny, nx, device=DEV, dtype=torch.bool)
    r = random.Random(seed)
    for _ in range(5):  # x-aligned high-permeability streaks, 8 cells wide and 4 high
        j, k = r.randrange(max(1, ny - 7)), r.randrange(max(1, nz - 3))
        streaks[k:k + 4, j:j + 8] = True
    lnk[streaks] += math.log(100.0)
    return lnk


def _cut(s):
    """Slices of [nz, ny, nx] for the cells that have the neighbour in slot s, and for those neighbours."""
    one = {0: (slice(None), slice(None)), 1: (slice(None, -1), slice(1, None)), -1: (slice(1, None), slice(None, -1))}
    di, dj, dk = SLOTS[s]
    own, other = zip(one[dk], one[dj], one[di])
    return own, other


def _blocks(nx, ny, nz, perm, seed):
    """The Jacobian as 3x3 blocks per cell and slot, [nz, ny, nx, 7, 3, 3] (absent faces zero), FP64."""
    g = _generator(seed)
    k = _permeability(nx, ny, nz, perm, g, seed).exp()
    a = torch.zeros(nz, ny, nx, 7, 3, 3, device=DEV, dtype=torch.float64)
    for s in (0, 1, 2, 4, 5, 6):
        own, other = _cut(s)
        t = 2.0 * k[own] * k[other] / (k[own] + k[other])
        m = 0.1 + 0.9 * torch.rand(*t.shape, 3, 3, device=DEV, dtype=torch.float64, generator=g)
        m.diagonal(dim1=-2, dim2=-1).add_(m.sum(-1))
        m *= t[..., None, None]
        a[own][..., s, :, :] = -m
        a[own][..., 3, :, :] += m
    acc = 0.2 * (1.0 + 4.0 * torch.rand(nz, ny, nx, 3, device=DEV, dtype=torch.float64, generator=g))
    a[..., 3, :, :].diagonal(dim1=-2, dim2=-1).add_(acc)
    return a


def _values(a):
    """The BSR values [nnzb, 3, 3] of the blocks: row by row, columns ascending, absent faces left out."""
    nz, ny, nx = a.shape[:3]
    has = torch.zeros(nz, ny, nx, 7, device=DEV, dtype=torch.bool)
    for s in range(7):
        has[_cut(s)[0]][..., s] = True
    return a[has]


def _rhs(cells, seed):
    """White noise plus a pair of wells on the pressure equation."""
    b = torch.randn(3 * cells, device=DEV, dtype=torch.float64, generator=_generator(seed + 7919))
    b[0] += 1e3
    b[3 * cells - 3] -= 1e3
    return b


def _vector(n, dtype, seed):
    return torch.randn(n, device=DEV, dtype=torch.float64, generator=_generator(seed + 104729)).to(dtype)


def _conv_inputs(case, seed):
    """Channels-last activations, weights [co][27][ci] (He-normal), bias and output gradient, as a layer meets them."""
    g = _generator(seed)
    v, ci, co = case["nx"] * case["ny"] * case["nz"], case["ci"], case["co"]
    x = torch.randn(v, ci, device=DEV, generator=g).clamp_(min=0).to(torch.bfloat16)
    w = (torch.randn(co, 27, ci, device=DEV, generator=g) * math.sqrt(2.0 / (27 * ci))).to(torch.bfloat16)
    bias = torch.randn(co, device=DEV, generator=g) * 0.1
    gy = (torch.randn(v, co, device=DEV, generator=g) / v ** 0.5).to(torch.bfloat16)
    return x, w, bias, gy


def _addr(t):
    return ctypes.c_void_p(t.data_ptr())


# ------------------------------------------------------------------ one case

def prepare(case, seed):
    kind = case["kind"]
    if kind == "conv":
        x, w, bias, gy = _conv_inputs(case, seed)
        st = dict(case=case, x=x, w=w, bias=bias, gy=gy)
        if case["direction"] == "forward":
            st["y"] = torch.empty_like(gy)
        else:
            st["gx"], st["gw"], st["gb"] = torch.empty_like(x), torch.empty(w.shape, device=DEV), torch.empty_like(bias)
        return st
    if kind == "batch":
        dims = _ensemble(case)
        A = rsv.Matrix.batch(dims)
        A.set_values(torch.cat([_values(_blocks(*d, "lognormal", seed + 31 * q)) for q, d in enumerate(dims)]))
        s = rsv.Solver(A, solver="bicgstab", rtol=TIGHT, precision=case["prec"])
        s.setup(case["pc"])
        b = torch.cat([_rhs(d[0] * d[1] * d[2], seed + 31 * q) for q, d in enumerate(dims)])
        return dict(case=case, A=A, s=s, b=b, x=torch.zeros_like(b))
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    A = rsv.Matrix(nx, ny, nz, precision=case["prec"])
    vals = _values(_blocks(nx, ny, nz, case["perm"], seed))
    A.set_values(vals)
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    st = dict(case=case, A=A, r=_vector(A.n, dtype, seed))
    st["z"] = torch.empty_like(st["r"])
    if kind == "spmv":
        return st
    if kind == "newton":
        st["vals"] = vals
    if kind in ("apply", "newton"):
        st["s"] = rsv.Solver(A, solver="gmres", restart=CYCLE, precision=case["prec"])
    elif kind == "cycle":
        st["s"] = rsv.Solver(A, solver="gmres", restart=CYCLE, rtol=0.0, maxit=CYCLE, precision=case["prec"])
    else:
        st["s"] = rsv.Solver(A, solver="gmres", restart=CYCLE, rtol=TIGHT, precision=case["prec"])
    st["s"].setup(case["pc"])
    if kind in ("cycle", "solve"):
        st["b"] = _rhs(A.nb, seed)
        st["x"] = torch.zeros_like(st["b"])
    return st


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "spmv":
        return state["A"].spmv(state["r"], state["z"])
    if kind == "apply":
        return state["s"].apply(state["r"], state["z"])
    if kind == "newton":
        state["A"].set_values(state["vals"])
        state["s"].setup(case["pc"])
        return state["s"].apply(state["r"], state["z"])
    if kind in ("cycle", "solve"):
        status, info = state["s"].solve(state["b"], state["x"].zero_())
        return dict(x=state["x"], status=status)
    if kind == "batch":
        status, info = state["s"].solve_batched(state["b"], state["x"].zero_())
        return dict(x=state["x"], status=status)
    nx, ny, nz, ci, co = (case[k] for k in ("nx", "ny", "nz", "ci", "co"))
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    x, w, bias, gy = state["x"], state["w"], state["bias"], state["gy"]
    if case["direction"] == "forward":
        rsv.check(rsv.rsv_conv3d_fwd(stream, nx, ny, nz, 27, ci, co, _addr(x), ci, _addr(w), _addr(bias), 1, None, 0,
                                     _addr(state["y"]), co, None))
        return state["y"]
    gx, gw, gb = state["gx"], state["gw"], state["gb"]
    # the layer's input came out of a ReLU: its gradient is masked by it
    rsv.check(rsv.rsv_conv3d_dgrad(stream, nx, ny, nz, ci, co, _addr(gy), co, _addr(w), _addr(x), ci, _addr(gx), ci,
                                   None))
    rsv.check(rsv.rsv_conv3d_wgrad(stream, nx, ny, nz, 27, ci, co, _addr(x), ci, _addr(gy), co, _addr(gw), _addr(gb)))
    return dict(gx=gx, gw=gw, gb=gb)


# ------------------------------------------------------------------ the least work

def _grid_work(nx, ny, nz, size):
    """(cells, blocks, one matrix read, one vector) in counts and bytes."""
    nb = nx * ny * nz
    nnzb = 7 * nb - 2 * (nx * ny + ny * nz + nx * nz)
    return nb, nnzb, 9 * size * nnzb, 3 * size * nb


def _spmv_work(nx, ny, nz, size):
    nb, nnzb, mat, vec = _grid_work(nx, ny, nz, size)
    return mat + 4 * (nnzb + nb) + 2 * vec, 18 * nnzb


def _apply_work(nx, ny, nz, size, pc):
    """ILU(0): off-diagonal blocks once, D^-1 in both sweeps, input and output.  A pressure stage adds its restriction,
    one V-cycle (five passes over the seven-point stencils of all levels, 8/7 of the finest) and, between two stages, a
    residual: from the pressure columns alone before a full stage that follows a first pressure stage, else whole."""
    nb, nnzb, mat, vec = _grid_work(nx, ny, nz, size)
    by, fl = 0, 0
    for q, stage in enumerate(STAGES[pc]):
        if stage == "F":
            by, fl = by + 9 * size * (nnzb - nb) + 18 * size * nb + 4 * vec, fl + 18 * (nnzb + nb)
        else:
            by, fl = by + 2 * vec + 8 / 7 * size * nb * (5 * 7 + 10), fl + 8 / 7 * nb * 5 * 14
        if q and STAGES[pc][:q] == "P":
            by, fl = by + mat / 3 + 2 * vec, fl + 6 * nnzb
        elif q:
            sb, sf = _spmv_work(nx, ny, nz, size)
            by, fl = by + sb + vec, fl + sf
    return by, fl


def _gmres_work(nx, ny, nz, size, pc, steps):
    """Per step: an application, a product, and the basis (15.5 vectors on average) read twice."""
    vec = _grid_work(nx, ny, nz, size)[3]
    sb, sf = _spmv_work(nx, ny, nz, size)
    pb, pf = _apply_work(nx, ny, nz, size, pc)
    return steps * (sb + pb + 33 * vec), steps * (sf + pf + 4 * 15.5 * vec / size)


def work(case):
    kind = case["kind"]
    if kind == "conv":
        v, ci, co = case["nx"] * case["ny"] * case["nz"], case["ci"], case["co"]
        one = 2 * v * 27 * ci * co
        if case["direction"] == "forward":
            return dict(bytes=2 * v * (ci + co) + 54 * ci * co, flops=one)
        return dict(bytes=2 * v * (2 * ci + co) + 54 * ci * co + 108 * ci * co, flops=2 * one)
    size = 8 if case["prec"] == "fp64" else 4
    if kind == "batch":  # some 200 passes of two applications and two products
        by = fl = 0
        for d in _ensemble(case):
            sb, sf = _spmv_work(*d, size)
            pb, pf = _apply_work(*d, size, "bilu0")
            by, fl = by + 200 * 2 * (sb + pb), fl + 200 * 2 * (sf + pf)
        return dict(bytes=by, flops=fl)
    d = case["nx"], case["ny"], case["nz"]
    if kind == "spmv":
        by, fl = _spmv_work(*d, size)
    elif kind == "apply":
        by, fl = _apply_work(*d, size, case["pc"])
    elif kind == "newton":  # values read, stored (and rounded), read for the factor, factor stored, applied
        nb, nnzb, mat, vec = _grid_work(*d, size)
        by, fl = _apply_work(*d, size, case["pc"])
        by, fl = by + 2 * 72 * nnzb + 3 * mat, fl + nb * 3 * 2 * 54
    elif kind == "cycle":
        by, fl = _gmres_work(*d, size, case["pc"], CYCLE)
    else:  # a tight solve of some 500 inner steps at half a million cells, growing with the grid's diameter
        by, fl = _gmres_work(*d, size, case["pc"], int(500 * (d[0] * d[1] * d[2] / 5e5) ** (1 / 3)) + 1)
    return dict(bytes=float(by), flops=float(fl))


# ------------------------------------------------------------------ 64-bit results, without the library

def _times(m, v):
    """3x3 blocks times 3-vectors, elementwise over the leading dimensions."""
    return (m * v[..., None, :]).sum(-1)


def _product(a, x):
    """A x for blocks a [nz, ny, nx, 7, 3, 3] and x [nz, ny, nx, 3]."""
    y = torch.zeros_like(x)
    for s in range(7):
        own, other = _cut(s)
        y[own] += _times(a[own][..., s, :, :], x[other])
    return y


class _Ilu0:
    """Block ILU(0) in natural order.  The seven-point graph has no triangles, so only the diagonal blocks change, and
    every cell of a plane i + j + k depends on the planes before it alone."""

    def __init__(self, a):
        nz, ny, nx = a.shape[:3]
        self.shape, nb = (nz, ny, nx), nx * ny * nz
        c = torch.arange(nb, device=DEV)
        plane = c % nx + (c // nx) % ny + c // (nx * ny)
        order = torch.argsort(plane, stable=True)
        self.planes = torch.split(order, torch.bincount(plane).tolist())
        self.off = (nx * ny, nx, 1)
        self.a = a.view(nb, 7, 3, 3)
        self.dinv = torch.zeros(nb, 3, 3, device=DEV, dtype=torch.float64)
        for p in self.planes:
            d = self.a[p, 3]
            for q in range(3):  # -z, -y, -x and, in that neighbour's row, the mirrored slot
                n = (p - self.off[q]).clamp_(min=0)  # an absent face has a zero block
                d = d - self.a[p, q] @ self.dinv[n] @ self.a[n, 6 - q]
            self.dinv[p] = torch.linalg.inv(d)

    def __call__(self, r):
        r = r.reshape(-1, 3)
        last = r.shape[0] - 1
        y, z = torch.zeros_like(r), torch.zeros_like(r)
        for p in self.planes:
            t = r[p]
            for q in range(3):
                t = t - _times(self.a[p, q], y[(p - self.off[q]).clamp_(min=0)])
            y[p] = _times(self.dinv[p], t)
        for p in reversed(self.planes):
            t = torch.zeros_like(y[p])
            for q in range(3):
                t = t + _times(self.a[p, 6 - q], z[(p + self.off[q]).clamp_(max=last)])
            z[p] = y[p] - _times(self.dinv[p], t)
        return z.view(*self.shape, 3)


class _Pressure:
    """Quasi-IMPES weights and one geometric V-cycle (2x2x2 boxes, piecewise-constant P, red-black Gauss-Seidel)."""

    def __init__(self, a, levels=6, coarse=512, sweeps=2):
        d = a[..., 3, :, :]
        self.w = torch.stack([torch.ones_like(d[..., 0, 0]), -d[..., 0, 1] / d[..., 1, 1], -d[..., 0, 2] / d[..., 2, 2]], -1)
        self.sweeps = sweeps
        self.ops = [(self.w[..., None, :, None] * a[..., :, :, :1]).sum((-1, -2)).movedim(-1, 0).contiguous()]
        while len(self.ops) < levels and self.ops[-1][0].numel() > coarse:
            self.ops.append(self._coarser(self.ops[-1]))
        last = self.ops[-1]
        n = last[0].numel()
        unit = torch.eye(n, device=DEV, dtype=torch.float64).view(n, *last.shape[1:])
        self.dense = torch.stack([self._stencil(last, e).reshape(-1) for e in unit], 1)
        self.colour = []
        for op in self.ops:
            k, j, i = (torch.arange(m, device=DEV) for m in op.shape[1:])
            self.colour.append((k[:, None, None] + j[None, :, None] + i[None, None, :]) % 2)

    @staticmethod
    def _coarser(op):
        nz, ny, nx = op.shape[1:]
        cz, cy, cx = (nz + 1) // 2, (ny + 1) // 2, (nx + 1) // 2
        f = torch.zeros(7, 2 * cz, 2 * cy, 2 * cx, device=DEV, dtype=torch.float64)
        f[:, :nz, :ny, :nx] = op
        f = f.view(7, cz, 2, cy, 2, cx, 2)
        out = torch.zeros(7, cz, cy, cx, device=DEV, dtype=torch.float64)
        out[3] = f[3].sum((1, 3, 5))
        for s, axis in ((0, 1), (1, 3), (2, 5), (4, 5), (5, 3), (6, 1)):
            inner, outer = (1, 0) if s < 3 else (0, 1)  # the child whose neighbour lies in the same box, or beyond it
            rest = tuple(x - (x > axis) for x in (1, 3, 5) if x != axis)
            out[3] += f[s].select(axis, inner).sum(rest)
            out[s] += f[s].select(axis, outer).sum(rest)
        return out

    @staticmethod
    def _stencil(op, x, diagonal=True):
        y = op[3] * x if diagonal else torch.zeros_like(x)
        for s in (0, 1, 2, 4, 5, 6):
            own, other = _cut(s)
            y[own] += op[s][own] * x[other]
        return y

    def _half(self, level, b, x, colour):
        op = self.ops[level]
        return torch.where(self.colour[level] == colour, (b - self._stencil(op, x, False)) / op[3], x)

    def _cycle(self, level, b):
        op = self.ops[level]
        if level + 1 == len(self.ops):
            return torch.linalg.solve(self.dense, b.reshape(-1)).view(b.shape)
        x = torch.zeros_like(b)
        for _ in range(self.sweeps):
            x = self._half(level, b, self._half(level, b, x, 0), 1)
        r = b - self._stencil(op, x)
        nz, ny, nx = r.shape
        cz, cy, cx = self.ops[level + 1].shape[1:]
        f = torch.zeros(2 * cz, 2 * cy, 2 * cx, device=DEV, dtype=torch.float64)
        f[:nz, :ny, :nx] = r
        e = self._cycle(level + 1, f.view(cz, 2, cy, 2, cx, 2).sum((1, 3, 5)))
        for axis in range(3):
            e = e.repeat_interleave(2, axis)
        x = x + e[:nz, :ny, :nx]
        for _ in range(self.sweeps):
            x = self._half(level, b, self._half(level, b, x, 1), 0)
        return x

    def __call__(self, r):
        x = torch.zeros_like(r)
        x[..., 0] = self._cycle(0, (self.w * r).sum(-1))
        return x


class _Preconditioner:
    """The stages of an order: the first acts on f, every later one on f - A x."""

    def __init__(self, a, pc):
        self.a, self.stages = a, STAGES[pc]
        self.of = {"F": _Ilu0(a)}
        if "P" in self.stages:
            self.of["P"] = _Pressure(a)

    def __call__(self, f):
        x = self.of[self.stages[0]](f)
        for stage in self.stages[1:]:
            x = x + self.of[stage](f - _product(self.a, x))
        return x


def _gmres_cycle(a, m, b, steps):
    """Right-preconditioned GMRES from zero: the minimal residual after `steps` steps (modified Gram-Schmidt, twice)."""
    beta = b.norm()
    v, z, h = [b / beta], [], torch.zeros(steps + 1, steps, device=DEV, dtype=torch.float64)
    for j in range(steps):
        z.append(m(v[j]))
        w = _product(a, z[j])
        for _ in range(2):
            for i, u in enumerate(v):
                t = (u * w).sum()
                h[i, j] += t
                w = w - t * u
        h[j + 1, j] = w.norm()
        v.append(w / h[j + 1, j])
    e = torch.zeros(steps + 1, 1, device=DEV, dtype=torch.float64)
    e[0] = beta
    y = torch.linalg.lstsq(h, e).solution[:, 0]
    return sum(t * u for t, u in zip(y, z))


def _exact_conv(case, seed):
    x, w, bias, gy = (t.double() for t in _conv_inputs(case, seed))
    nx, ny, nz, ci, co = (case[k] for k in ("nx", "ny", "nz", "ci", "co"))

    def shifted(t, c):  # the volume with a border of zeros, seen from each of the 27 taps
        p = torch.zeros(nz + 2, ny + 2, nx + 2, c, device=DEV, dtype=torch.float64)
        p[1:-1, 1:-1, 1:-1] = t.view(nz, ny, nx, c)
        return [p[q // 9:q // 9 + nz, q // 3 % 3:q // 3 % 3 + ny, q % 3:q % 3 + nx].reshape(-1, c) for q in range(27)]

    if case["direction"] == "forward":
        return (sum(t @ w[:, q].T for q, t in enumerate(shifted(x, ci))) + bias).clamp_(min=0)
    gx = sum(t @ w[:, 26 - q] for q, t in enumerate(shifted(gy, co)))
    gw = torch.stack([gy.T @ t for t in shifted(x, ci)], 1)
    return dict(gx=gx * (x > 0), gw=gw, gb=gy.sum(0))


def exact(case, seed):
    kind = case["kind"]
    if kind == "conv":
        return _exact_conv(case, seed)
    if kind in ("batch", "solve"):  # an iteration to a tolerance: what it returns depends on where it stops
        return None
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    if kind == "cycle" and nx * ny * nz > 100_000:
        return None
    a = _blocks(nx, ny, nz, case["perm"], seed)
    if kind == "cycle":
        b = _rhs(nx * ny * nz, seed).view(nz, ny, nx, 3)
        x = _gmres_cycle(a, _Preconditioner(a, case["pc"]), b, CYCLE)
        return dict(x=x.reshape(-1), status=None)
    dtype = torch.float64 if case["prec"] == "fp64" else torch.float32
    a = a.to(dtype).double()  # a mixed-precision solver works on the matrix rounded to FP32
    r = _vector(3 * nx * ny * nz, dtype, seed).double().view(nz, ny, nx, 3)
    z = _product(a, r) if kind == "spmv" else _Preconditioner(a, case["pc"])(r)
    return z.reshape(-1)
