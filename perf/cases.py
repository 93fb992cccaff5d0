"""The calls that a user of this library makes, at the sizes they are made at.

Each case is one call (or one short sequence of calls) of the public Python
binding on a start state that stays as it is: a pass copies the start state
into the buffers the library advances in place and calls it, so every pass
does the same work.  The start velocities are a discrete curl (divergence-free
to rounding) of a few smooth vortices plus small noise on the faces -- a flow
in motion, as every slice of a Parareal call after the first holds -- in a box
whose lid moves; pressures start at zero, as after a restart.

Kinds of case and what each stands for:
  step     time stepping of one state or a batch (the fine propagator)
  coarse   the serial coarse propagator: one state, large steps
  parareal a whole Parareal call
  graph    several independent cavities in one captured launch
  adjoint  value and gradient of the final kinetic energy through autograd
  poisson  the pressure solve on its own
  predict  the explicit part of a step on its own
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1705_06149_gb300 import Grid, State, StepGraph
from paper_1705_06149_gb300.autograd import kinetic_energy
from paper_1705_06149_gb300.inputs import mixed_batch_sizes, obstacle_boxes

WALLS = "wall,wall,wall"
DEV = torch.device("cuda")


def _case(name, kind, n, *, box=(1.0, 1.0, 1.0), bc=WALLS, prec="fp32_refine", batch=1, re=1000.0,
          dt=5e-4, steps=1, **more):
    c = dict(kind=kind, nx=n[0], ny=n[1], nz=n[2], lx=float(box[0]), ly=float(box[1]),
             lz=float(box[2]), bc=bc, prec=prec, batch=batch, re=re, dt=dt, steps=steps, **more)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # one step of the smallest cavity in FP64: the cost of a call
        _case("step_16_fp64", "step", (16, 16, 16), prec="fp64", re=100.0, dt=1e-3),
        # the plain method end to end: 16^3, Re 100, 4 slices of 50 steps, coarse step 10x,
        # 4 iterations, FP64
        _case("parareal_16_fp64", "parareal", (16, 16, 16), prec="fp64", re=100.0, dt=1e-3,
              batch=4, steps=50, coarse=5, iterations=4),
        # the fine sweep of the 64^3 cavity: 32 slices in one call
        _case("sweep_64x32_fp32", "step", (64, 64, 64), batch=32, steps=10),
        # Parareal on the 64^3 cavity with 32 slices (shorter slices than a production run)
        _case("parareal_64x32_fp32", "parareal", (64, 64, 64), batch=32, steps=10, coarse=1,
              iterations=2),
        # the coarse propagator of that cavity: serial steps of one state
        _case("coarse_64_fp32", "coarse", (64, 64, 64), dt=5e-3, steps=5),
        # the same cavity in FP64, a few slices
        _case("sweep_64x4_fp64", "step", (64, 64, 64), prec="fp64", batch=4, steps=4),
        # the largest grid of the mixed batch, a few of its slices
        _case("sweep_256x4_fp32", "step", (256, 256, 256), batch=4, steps=2),
        # a cavity with solid boxes
        _case("obstacles_128x8_fp32", "step", (128, 128, 128), batch=8, steps=2, boxes=8),
        # independent cavities of mixed sizes and Reynolds numbers in one graph launch
        _case("mixed_graph_fp32", "graph", (96, 96, 96), steps=5, cavities=6, pick=0),
        # gradient of the final kinetic energy on the 64^3 cavity
        _case("adjoint_64_fp32", "adjoint", (64, 64, 64), re=400.0, dt=1e-3, steps=20, ckpt=5),
        # odd sizes along every axis
        _case("step_odd_45_37_51_fp32", "step", (45, 37, 51), batch=3, steps=3),
        # the pressure solve alone, FP64, on a channel (periodic x, slip z)
        _case("poisson_96_64_48_fp64", "poisson", (96, 64, 48), box=(3.0, 2.0, 1.5),
              bc="periodic,wall,slip", prec="fp64", batch=4),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "coarse", "parareal", "graph", "adjoint",
                       "poisson", "predict"])
    prec = rng.choice(["fp32_refine", "fp32_refine", "fp64"])
    bc = ",".join(rng.choice(["wall", "wall", "periodic", "slip"]) for _ in range(3))
    # sizes: any, or multiples of 4, 8 or 16 (grids the hierarchy halves); the
    # box follows the cells up to a factor 2 per axis
    m = rng.choice([1, 4, 8, 16])
    top = {1: 64, 4: 96, 8: 160, 16: 192}[m]
    if prec == "fp64":
        top = min(top, 96)
    dims = [max(m, _log_int(rng, 12, top) // m * m) for _ in range(3)]
    while dims[0] * dims[1] * dims[2] > (1 << 18 if m == 1 else 1 << 22):
        dims[dims.index(max(dims))] = max(m, dims[dims.index(max(dims))] // 2 // m * m)
    dims = [max(4, d) for d in dims]
    box = [d / max(dims) * rng.uniform(0.7, 1.4) for d in dims]
    cells = dims[0] * dims[1] * dims[2]
    room = (1 << 22) if prec == "fp32_refine" else (1 << 20)
    dt = 0.03 / max(dims)
    batch = max(1, min(32, _log_int(rng, 1, 32), room // cells))
    kw = dict(box=box, bc=bc, prec=prec, re=round(rng.uniform(100.0, 2000.0), 1), dt=dt)
    if kind == "step":
        if rng.random() < 0.15 and min(dims) >= 24 and m >= 8:
            kw["boxes"] = rng.randint(1, 4 if min(dims) < 64 else 8)
            kw["box"] = (1.0, 1.0, 1.0)
        return _case(None, "step", dims, batch=batch, steps=rng.randint(1, 4), **kw)
    if kind == "coarse":
        kw["dt"] = 5 * dt
        return _case(None, "coarse", dims, steps=rng.randint(1, 5), **kw)
    if kind == "predict":
        return _case(None, "predict", dims, batch=batch, **kw)
    if kind == "poisson":
        return _case(None, "poisson", dims, batch=batch, **kw)
    if kind == "graph":
        return _case(None, "graph", (96, 96, 96), steps=rng.randint(1, 5),
                     cavities=rng.randint(1, 6), pick=rng.randint(0, 18), prec="fp32_refine",
                     dt=5e-4)
    if kind == "adjoint":
        dims = [max(8, d // 2) if d > 64 else d for d in dims]
        steps = max(2, min(10, (1 << 21) // (dims[0] * dims[1] * dims[2])))
        return _case(None, "adjoint", dims, steps=steps, ckpt=rng.randint(1, 6), **kw)
    dims = [min(d, 32 if m == 1 else 64) for d in dims]
    slices = rng.randint(2, 16)
    return _case(None, "parareal", dims, batch=slices, steps=rng.randint(2, 10), coarse=1,
                 iterations=rng.randint(1, 2), **kw)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _bc(case):
    return tuple(case["bc"].split(","))


def _dims(case):
    return (case["nx"], case["ny"], case["nz"])


def _box(case):
    return (case["lx"], case["ly"], case["lz"])


def _extents(n, bc, c):
    """Stored positions of component c along x, y, z."""
    return [n[d] + (1 if d == c and bc[d] != "periodic" else 0) for d in range(3)]


def _axis(t, d):
    return t.dim() - 1 - d


def _velocity(n, box, bc, batch, seed, solid=None):
    """u, v, w in FP64: the discrete curl of a random smooth edge potential
    (zero on walls) plus N(0, 1e-3^2) on every moving face."""
    dev = DEV
    gen = torch.Generator(device=dev).manual_seed(seed)
    pot = []
    for a in range(3):  # component a of the potential lives on edges along a
        ext = [n[d] if d == a else n[d] + 1 for d in range(3)]
        total = torch.zeros([batch] + ext[::-1], dtype=torch.float64, device=dev)
        for mode in (1, 2, 3):
            amp = torch.randn(batch, 1, 1, 1, dtype=torch.float64, device=dev, generator=gen)
            shape = torch.ones([1, 1, 1, 1], dtype=torch.float64, device=dev)
            for d in range(3):
                x = torch.arange(ext[d], dtype=torch.float64, device=dev)
                if d == a:
                    f = torch.cos(math.pi * (mode - 1) * (x + 0.5) / n[d] * (
                        2 if bc[d] == "periodic" else 1))
                elif bc[d] == "periodic":
                    f = torch.sin(2 * math.pi * mode * x / n[d])
                else:
                    f = torch.sin(math.pi * mode * x / n[d])
                    f[0] = 0.0
                    f[-1] = 0.0
                view = [1, 1, 1, 1]
                view[3 - d] = ext[d]
                shape = shape * f.view(view)
            total = total + amp / mode * shape
        pot.append(total * (0.05 * min(box)))
    h = [box[d] / n[d] for d in range(3)]
    vel = []
    for c in range(3):
        a, b = (c + 1) % 3, (c + 2) % 3
        f = (torch.diff(pot[b], dim=_axis(pot[b], a)) / h[a]
             - torch.diff(pot[a], dim=_axis(pot[a], b)) / h[b])
        if bc[c] == "periodic":
            f = f.narrow(_axis(f, c), 0, n[c])
        vel.append(f.contiguous())
    act = _active(n, bc, solid, dev)
    for c in range(3):
        noise = torch.randn(vel[c].shape, dtype=torch.float64, device=dev, generator=gen)
        vel[c] = (vel[c] + 1e-3 * noise) * act[c]
    return vel


def _solid(case, seed=0):
    if not case.get("boxes"):
        return None
    # the boxes belong to the workload, not to the state: the same for every seed
    return obstacle_boxes(_dims(case), seed=seed, count=case["boxes"], edge=(0.08, 0.2))[1]


def _cavities(case):
    dims, res = mixed_batch_sizes(24, seed=0)
    return [(dims[q], res[q]) for q in range(case["pick"], case["pick"] + case["cavities"])]


def _start(case, seed):
    """The start state(s) as lists [u, v, w, p] of device tensors in the grid's types."""
    bc = _bc(case)
    vt = torch.float32 if case["prec"] == "fp32_refine" else torch.float64
    if case["kind"] == "graph":
        out = []
        for q, (n, _) in enumerate(_cavities(case)):
            vel = _velocity(n, _box(case), bc, 1, 100 * seed + q)
            out.append([t.to(vt) for t in vel] + [torch.zeros((1,) + n[::-1], dtype=torch.float64,
                                                              device=DEV)])
        return out
    n = _dims(case)
    solid = _solid(case)
    batch = 1 if case["kind"] == "parareal" else case["batch"]
    vel = _velocity(n, _box(case), bc, batch, seed, solid)
    p = torch.zeros((batch,) + n[::-1], dtype=torch.float64, device=DEV)
    return [t.to(vt).contiguous() for t in vel] + [p]


def _rhs(case, seed):
    """Right sides of the pressure solve: a divergence's spectrum (rough) over smooth modes."""
    n = _dims(case)
    gen = torch.Generator(device=DEV).manual_seed(seed)
    b = torch.randn((case["batch"],) + n[::-1], dtype=torch.float64, device=DEV, generator=gen)
    for d in range(3):
        x = (torch.arange(n[d], dtype=torch.float64, device=DEV) + 0.5) / n[d]
        view = [1, 1, 1, 1]
        view[3 - d] = n[d]
        b = b + 3.0 * torch.cos(2 * math.pi * (d + 1) * x).view(view)
    return b.contiguous()


def _grid(case, n=None, re=None, batch=None):
    n = n or _dims(case)
    return Grid(*n, *_box(case), re=re or case["re"], u_lid=1.0, bc=_bc(case),
                precision=case["prec"], batch=batch or case["batch"], solid=_solid(case))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        b = _rhs(case, seed)
        return {"case": case, "grid": _grid(case), "b": b, "p": torch.zeros_like(b)}
    start = _start(case, seed)
    if kind == "graph":
        grids = [_grid(case, n, re) for n, re in _cavities(case)]
        work = [State(*[t.clone() for t in st]) for st in start]
        graph = StepGraph([(g, w, case["dt"], case["steps"]) for g, w in zip(grids, work)])
        return {"case": case, "grids": grids, "start": start, "work": work, "graph": graph}
    g = _grid(case)
    s = {"case": case, "grid": g, "start": State(*start)}
    if kind == "parareal":
        s["slices"] = g.zeros(case["batch"] + 1)
    elif kind == "adjoint":
        s["leaves"] = [t.requires_grad_(True) for t in start[:3]]
        s["lid"] = torch.tensor(1.0, dtype=torch.float64, requires_grad=True)
    elif kind != "predict":
        s["work"] = s["start"].clone()
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "poisson":
        state["p"].zero_()
        state["grid"].poisson_solve(state["b"], state["p"])
        return state["p"]
    if kind == "graph":
        for src, dst in zip(state["start"], state["work"]):
            for a, b in zip(src, dst.fields()):
                b.copy_(a)
        state["graph"].launch()
        state["graph"].check()
        return [w.fields() for w in state["work"]]
    g = state["grid"]
    if kind == "parareal":
        _, defects = g.parareal(state["start"], state["slices"], case["batch"], case["steps"],
                                case["coarse"], case["dt"], case["iterations"])
        return [state["slices"].fields(), torch.tensor(defects, dtype=torch.float64)]
    if kind == "adjoint":
        u, v, w = state["leaves"]
        J = kinetic_energy(u, v, w, state["lid"], g, case["dt"], case["steps"], case["ckpt"])
        grads = torch.autograd.grad(J.sum(), [u, v, w, state["lid"]])
        return [J.detach(), list(grads)]
    if kind == "predict":
        return list(g.predict(state["start"], case["dt"]))
    work = state["work"]
    for a, b in zip(state["start"].fields(), work.fields()):
        b.copy_(a)
    if kind == "coarse":
        g.step_coarse(work, case["dt"], case["steps"])
    else:
        g.step_fine(work, case["dt"], case["steps"])
    return work.fields()


# ---------------------------------------------------------------------------
# work and tolerance
# ---------------------------------------------------------------------------

# Operations per cell and step: six upwind fluxes and three second differences
# for each of three components (about 250), divergence, gradient and
# correction (about 30), and a pressure solve (at least about 100: two
# residuals, a correction and their norms).
STEP_FLOPS = 400.0


def work(case):
    """A step reads and writes a state (three velocity components and the
    FP64 pressure); nothing else has to leave the chip."""
    cells = float(case["nx"] * case["ny"] * case["nz"])
    vb = 4.0 if case["prec"] == "fp32_refine" else 8.0
    state = 3.0 * vb + 8.0
    kind = case["kind"]
    if kind == "poisson":
        return {"bytes": 24.0 * cells * case["batch"], "flops": 100.0 * cells * case["batch"]}
    if kind == "predict":
        return {"bytes": 6.0 * vb * cells * case["batch"], "flops": 250.0 * cells * case["batch"]}
    if kind == "graph":
        total = float(sum(n[0] * n[1] * n[2] for n, _ in _cavities(case)))
        cell_steps = total * case["steps"]
    elif kind == "parareal":
        k, s, m = case["iterations"], case["steps"], case["coarse"]
        cell_steps = cells * case["batch"] * (k * s + (k + 1) * m)
    elif kind == "adjoint":
        # forward, recomputation from the checkpoints, reverse
        cell_steps = 3.0 * cells * case["batch"] * case["steps"]
    else:
        cell_steps = cells * case["batch"] * case["steps"]
    return {"bytes": 2.0 * state * cell_steps, "flops": STEP_FLOPS * cell_steps}


def tolerance(case):
    """About four times the largest error against exact() that was measured."""
    if case["prec"] == "fp64":
        # solves stop at a relative residual of 1e-12; a pressure carries that
        # times the conditioning of the operator (up to 1.7e-10 measured on an
        # odd grid, 4e-13 in steps)
        return {"rel": 2e-14 if case["kind"] == "predict" else 1e-9}
    if case["kind"] == "predict":
        return {"rel": 1e-7}  # 2.5e-8 measured
    if case["kind"] == "adjoint":
        # SMART's derivative jumps where a face changes its branch: faces within
        # FP32 rounding of a branch point take either (2.9e-6 measured)
        return {"rel": 2e-5}
    # FP32 storage of the velocity; a pressure is its divergence over dt, and a
    # Parareal update adds the difference of two coarse values (8.4e-7 measured)
    return {"rel": 5e-6}


# ---------------------------------------------------------------------------
# the same in plain torch, FP64
# ---------------------------------------------------------------------------

def _active(n, bc, solid, dev):
    """Faces that move: not a wall-normal boundary face, no solid neighbour."""
    out = []
    fluid = None
    if solid is not None:
        fluid = torch.as_tensor(np.asarray(solid) == 0, device=dev)
    for c in range(3):
        ext = _extents(n, bc, c)
        m = torch.ones(ext[::-1], dtype=torch.bool, device=dev)
        ax = 2 - c
        if bc[c] != "periodic":
            m.select(ax, 0).fill_(False)
            m.select(ax, ext[c] - 1).fill_(False)
        if fluid is not None:
            if bc[c] == "periodic":
                both = fluid & torch.roll(fluid, 1, ax)
                m = m & both
            else:
                inner = fluid.narrow(ax, 0, n[c] - 1) & fluid.narrow(ax, 1, n[c] - 1)
                m.narrow(ax, 1, n[c] - 1).logical_and_(inner)
        out.append(m)
    return out


class _Reference:
    """One grid of the scheme in FP64: ghost values, SMART convection, the
    pressure equation solved through the eigenvectors of its three 1D
    operators (with solid cells: conjugate gradients preconditioned by that)."""

    def __init__(self, case, n=None, re=None):
        self.n = n or _dims(case)
        self.bc = _bc(case)
        self.dev = DEV
        box = _box(case)
        self.h = [box[d] / self.n[d] for d in range(3)]
        self.re = re or case["re"]
        self.lid = torch.tensor(1.0, dtype=torch.float64, device=self.dev)
        solid = _solid(case)
        self.act = _active(self.n, self.bc, solid, self.dev)
        self.fluid = None
        if solid is not None:
            self.fluid = torch.as_tensor(np.asarray(solid) == 0, device=self.dev)
            self.in_solid = self._faces_in_solid()
        self.q, lam = [], []
        for d in range(3):
            m = self.n[d]
            a = np.zeros((m, m))
            for i in range(m):
                for j in (i - 1, i + 1):
                    if 0 <= j < m or self.bc[d] == "periodic":
                        a[i, j % m] += 1.0
                        a[i, i] -= 1.0
            w, v = np.linalg.eigh(a)
            self.q.append(torch.as_tensor(v, device=self.dev))
            lam.append(torch.as_tensor(w / self.h[d] ** 2, device=self.dev))
        s = lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
        s.view(-1)[torch.argmax(s)] = float("inf")  # the constant
        self.inv = 1.0 / s

    def _faces_in_solid(self):
        out = []
        for c in range(3):
            ax = 2 - c
            s = ~self.fluid
            if self.bc[c] == "periodic":
                out.append(s & torch.roll(s, 1, ax))
            else:
                m = torch.zeros(_extents(self.n, self.bc, c)[::-1], dtype=torch.bool,
                                device=self.dev)
                m.narrow(ax, 1, self.n[c] - 1).copy_(
                    s.narrow(ax, 0, self.n[c] - 1) & s.narrow(ax, 1, self.n[c] - 1))
                out.append(m)
        return out

    # --- ghosts -----------------------------------------------------------
    def pad(self, c, a):
        for d in range(3):
            ax = _axis(a, d)
            e = a.shape[ax]

            def at(i):
                return a.narrow(ax, i, 1)

            if self.bc[d] == "periodic":
                lo, hi = [at((e - 2) % e), at(e - 1)], [at(0), at(1 % e)]
            elif d == c:
                lo, hi = [-at(2), -at(1)], [-at(e - 2), -at(e - 3)]
            else:
                s = 1.0 if self.bc[d] == "slip" else -1.0
                add = 2.0 * self.lid if c == 0 and d == 1 and self.bc[d] == "wall" else 0.0
                lo, hi = [s * at(1), s * at(0)], [add + s * at(e - 1), add + s * at(e - 2)]
            a = torch.cat(lo + [a] + hi, dim=ax)
        return a

    def _win(self, padded, ext, off):
        """Values at offset off from each of the first ext positions."""
        out = padded
        for d in range(3):
            out = out.narrow(_axis(out, d), 2 + off[d], ext[d])
        return out

    def _mask_at(self, mask, d, m, c):
        """mask of component c's positions, shifted by m along axis d (False outside)."""
        ax = 2 - d
        if self.bc[d] == "periodic":
            return torch.roll(mask, -m, ax)
        out = torch.zeros_like(mask)
        e = mask.shape[ax]
        k = e - abs(m)
        if k > 0:
            out.narrow(ax, max(0, -m), k).copy_(mask.narrow(ax, max(0, m), k))
        return out

    def arms(self, c, d, padded):
        """The five values along axis d that a face of component c sees: past the
        first solid surface the arm is reflected like at a wall."""
        ext = _extents(self.n, self.bc, c)

        def val(m):
            off = [0, 0, 0]
            off[d] = m
            return self._win(padded, ext, off)

        a = {m: val(m) for m in range(-2, 3)}
        if self.fluid is None:
            return [a[m] for m in range(-2, 3)]
        out = dict(a)
        for s in (-1, 1):
            if c == d:
                idle = ~self.act[c]
                s1, s2 = self._mask_at(idle, d, s, c), self._mask_at(idle, d, 2 * s, c)
                out[s] = torch.where(s1, torch.zeros_like(a[0]), a[s])
                out[2 * s] = torch.where(s1, -a[0], torch.where(s2, torch.zeros_like(a[0]),
                                                                a[2 * s]))
            else:
                sol = self.in_solid[c]
                s1, s2 = self._mask_at(sol, d, s, c), self._mask_at(sol, d, 2 * s, c)
                out[s] = torch.where(s1, -a[0], a[s])
                # past a wall the ghost is the mirror of its own image, solid or not
                ax = 2 - d
                pos = torch.arange(ext[d], device=self.dev)
                beyond = (pos + s < 0) | (pos + s >= ext[d])
                if self.bc[d] == "periodic":
                    beyond = torch.zeros_like(beyond)
                view = [1, 1, 1]
                view[ax] = ext[d]
                s1 = s1 & ~beyond.view(view)
                out[2 * s] = torch.where(s1, -a[-s], torch.where(s2, -a[s], a[2 * s]))
        return [out[m] for m in range(-2, 3)]

    # --- the explicit part --------------------------------------------------
    @staticmethod
    def _smart(uf, bb, b, f, ff):
        pos = uf > 0
        U, C, D = torch.where(pos, bb, ff), torch.where(pos, b, f), torch.where(pos, f, b)
        cc, dd = C - U, D - U
        a = torch.where(dd > 0, cc, -cc)
        r = dd.abs()
        phi = torch.where(6 * a <= r, U + 3 * cc,
                          torch.where(6 * a <= 5 * r, U + 0.75 * cc + 0.375 * dd, D))
        phi = torch.where((dd == 0) | (a < 0) | (a > r), C, phi)
        return uf * phi

    def predict(self, vel, dt):
        pads = [self.pad(c, vel[c]) for c in range(3)]
        out = []
        for c in range(3):
            ext = _extents(self.n, self.bc, c)
            rhs = 0.0
            for d in range(3):
                a0, a1, a2, a3, a4 = self.arms(c, d, pads[c])
                if d == c:
                    up, um = 0.5 * (a2 + a3), 0.5 * (a1 + a2)
                else:
                    def tr(oc, od):
                        off = [0, 0, 0]
                        off[c], off[d] = oc, od
                        return self._win(pads[d], ext, off)
                    up = 0.5 * (tr(-1, 1) + tr(0, 1))
                    um = 0.5 * (tr(-1, 0) + tr(0, 0))
                conv = (self._smart(up, a1, a2, a3, a4) - self._smart(um, a0, a1, a2, a3))
                rhs = rhs + (a3 - 2 * a2 + a1) / (self.re * self.h[d] ** 2) - conv / self.h[d]
            out.append(torch.where(self.act[c], vel[c] + dt * rhs, torch.zeros_like(vel[c])))
        return out

    # --- the projection -------------------------------------------------------
    def div(self, f):
        out = 0.0
        for d in range(3):
            ax = _axis(f[d], d)
            hi = torch.roll(f[d], -1, ax) if self.bc[d] == "periodic" else f[d].narrow(ax, 1, self.n[d])
            out = out + (hi - f[d].narrow(ax, 0, self.n[d])) / self.h[d]
        return out

    def grad(self, p):
        out = []
        for d in range(3):
            ax = _axis(p, d)
            if self.bc[d] == "periodic":
                g = (p - torch.roll(p, 1, ax)) / self.h[d]
            else:
                inner = torch.diff(p, dim=ax) / self.h[d]
                z = torch.zeros_like(p.narrow(ax, 0, 1))
                g = torch.cat([z, inner, z], dim=ax)
            out.append(torch.where(self.act[d], g, torch.zeros_like(g)))
        return out

    def lap(self, p):
        return self.div(self.grad(p))

    def box_solve(self, b):
        q = self.q
        x = torch.matmul(b, q[0])
        x = torch.matmul(q[1].T, x)
        x = torch.einsum("zk,bzyx->bkyx", q[2], x) * self.inv
        x = torch.einsum("zk,bkyx->bzyx", q[2], x)
        return torch.matmul(torch.matmul(q[1], x), q[0].T)

    def mean_free(self, p):
        if self.fluid is None:
            return p - p.mean(dim=(1, 2, 3), keepdim=True)
        m = p.masked_fill(~self.fluid, 0.0)
        return (m - m.sum(dim=(1, 2, 3), keepdim=True) / self.fluid.sum()).masked_fill(
            ~self.fluid, 0.0)

    def solve(self, b):
        b = self.mean_free(b)
        if self.fluid is None:
            x = self.box_solve(b)
            x = x + self.box_solve(b - self.lap(x))
            return self.mean_free(x)

        def dot(a, c):
            return (a * c).sum(dim=(1, 2, 3), keepdim=True)

        x = torch.zeros_like(b)
        r = b.clone()
        z = self.mean_free(self.box_solve(r))
        p = z
        rz = dot(r, z)
        bb = dot(b, b)
        for _ in range(300):
            ap = self.lap(p)
            alpha = rz / dot(p, ap)
            x = x + alpha * p
            r = r - alpha * ap
            if bool((dot(r, r) <= 1e-27 * bb).all()):
                break
            z = self.mean_free(self.box_solve(r))
            rz1 = dot(r, z)
            p = z + (rz1 / rz) * p
            rz = rz1
        return self.mean_free(x)

    def step(self, vel, dt, steps):
        p = None
        for _ in range(steps):
            f = self.predict(vel, dt)
            p = self.solve(self.div(f) / dt)
            vel = [a - dt * g for a, g in zip(f, self.grad(p))]
        return vel, p


def _exact_parareal(case, vel):
    ref = _Reference(case)
    n_sl, S, M, dt = case["batch"], case["steps"], case["coarse"], case["dt"]
    dtc = dt * S / M

    def coarse(y):
        v, p = ref.step(y[:3], dtc, M)
        return v + [p]

    y = [vel + [torch.zeros((1,) + _dims(case)[::-1], dtype=torch.float64, device=DEV)]]
    g_old = []
    for k in range(n_sl):
        g_old.append(coarse(y[k]))
        y.append(g_old[k])
    defects = []
    for _ in range(case["iterations"]):
        v, p = ref.step([torch.cat([y[k][c] for k in range(n_sl)]) for c in range(3)], dt, S)
        fine = v + [p]
        new = [y[0]]
        worst = 0.0
        for k in range(n_sl):
            g = coarse(new[k])
            nxt = [fine[c][k:k + 1] + (g[c] - g_old[k][c]) for c in range(4)]
            worst = max([worst] + [float((nxt[c] - y[k + 1][c]).abs().max()) for c in range(4)])
            g_old[k] = g
            new.append(nxt)
        y = new
        defects.append(worst)
    return [[torch.cat([y[k][c] for k in range(n_sl + 1)]) for c in range(4)],
            torch.tensor(defects, dtype=torch.float64)]


def exact(case, seed):
    kind = case["kind"]
    if kind == "poisson":
        with torch.no_grad():
            return _Reference(case).solve(_rhs(case, seed))
    start = _start(case, seed)
    if kind == "graph":
        out = []
        with torch.no_grad():
            for (n, re), st in zip(_cavities(case), start):
                v, p = _Reference(case, n, re).step([t.double() for t in st[:3]], case["dt"],
                                                    case["steps"])
                out.append(v + [p])
        return out
    vel = [t.double() for t in start[:3]]
    if kind == "adjoint":
        ref = _Reference(case)
        vel = [t.requires_grad_(True) for t in vel]
        ref.lid = ref.lid.clone().requires_grad_(True)
        # every active face of the start is a variable; inactive ones hold zero
        v, _ = ref.step([torch.where(m, t, torch.zeros_like(t)) for m, t in zip(ref.act, vel)],
                        case["dt"], case["steps"])
        vol = ref.h[0] * ref.h[1] * ref.h[2]
        J = sum(0.5 * vol * (t * t).sum(dim=(1, 2, 3)) for t in v)
        grads = torch.autograd.grad(J.sum(), vel + [ref.lid])
        if case["prec"] != "fp64":
            # the branch an FP32 trajectory takes next to a branch point decides
            # the derivative there: no one gradient of 64 bits belongs to it
            grads = [None, None, None, grads[3]]
        return [J.detach(), list(grads)]
    with torch.no_grad():
        if kind == "parareal":
            return _exact_parareal(case, vel)
        ref = _Reference(case)
        if kind == "predict":
            return ref.predict(vel, case["dt"])
        v, p = ref.step(vel, case["dt"], case["steps"])
        return v + [p]
