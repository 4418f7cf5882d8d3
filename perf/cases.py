"""The work that a user has this framework do, as timed cases.

One case is one pass through the public entry points: set the fields, advance a
number of steps, take out what a program takes out (fields, Delta*, totals, the
state for a checkpoint, gradients).  The grids, velocity sets, step sizes and the
ensemble are those of ``workloads.py``, the tests and ``bench.py``; a pass runs a
share of their step counts.  The initial fields are theirs with amplitudes, phases
or left and right states drawn from the seed.
"""
import math

import numpy as np
import torch
import torch.utils.checkpoint

from paper_2502_16818_gb300 import BatchSolver, Solver, workloads as W
from paper_2502_16818_gb300.cdbm import make_run_function

PRECISIONS = {"fp64": 0, "bulk": 1, "df64": 2, "dev": 3}
FIELDS = ("rho", "ux", "uy", "T")


# ------------------------------------------------------------------ the cases

def listed():
    return [
        # a program that writes its fields after every step of a small square: launches and latency
        _case("square_64_each_step", "smooth", "fp64", 64, 64, 1, 1.0),
        # the Sod tube of Sec. 3.1, a twentieth of its 10^4 steps
        _case("sod_500", "sod", "fp64", 500, 1, 500, 0.0),
        # the Lax tube of Sec. 3.2, likewise
        _case("lax_2000", "lax", "fp64", 2000, 1, 500, 0.0),
        # the sound wave of Sec. 3.4 on 512^2: a state that the L2 cache holds
        _case("sound_512", "sound", "fp64", 512, 512, 50, 1.0),
        # the Taylor-Green vortex of Sec. 3.5 on 4096^2 in double: the headline run
        _case("vortex_4096", "vortex", "fp64", 4096, 4096, 10, 3.0),
        # the same vortex with the two fast single-precision equilibria
        _case("vortex_4096_df64", "vortex", "df64", 4096, 4096, 20, 3.0),
        _case("vortex_4096_dev", "vortex", "dev", 4096, 4096, 20, 3.0),
        # a ragged rectangle with zero-gradient edges in the double-equilibrium single-precision mode
        _case("smooth_1500x1300_bulk", "smooth", "bulk", 1500, 1300, 20, 1.0, bc=1),
        # Delta*, fields and totals of a resident state, as a program does when it writes a frame
        _case("frame_2048", "frame", "fp64", 2048, 2048, 4, 3.0),
        # the ensemble of shock tubes, in double and in double-float
        _case("ensemble_1024", "ensemble", "fp64", 1024, 4000, 100, 0.0),
        _case("ensemble_1024_df64", "ensemble", "df64", 1024, 4000, 200, 0.0),
        # gradients of a run through autograd: forward with checkpoints, then backward
        _case("adjoint_512", "adjoint", "fp64", 512, 512, 40, 3.0, every=20, limiter=2),
    ]


def _case(name, kind, precision, nx, ny, steps, I, bc=0, every=0, limiter=0):
    """nx, ny: cells (for the ensemble: tubes, and the longest tube's cells); every, limiter:
    checkpoint interval and limiter linearisation of the adjoint."""
    return {"name": name, "kind": kind, "precision": precision, "nx": nx, "ny": ny, "steps": steps, "I": I,
            "bc": bc, "every": every, "limiter": limiter}


def draw(rng):
    def size(lo, hi):
        n = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
        return n + 1 if rng.random() < 0.3 and n < hi else n

    kind = rng.choice(["sod", "lax", "sound", "vortex", "vortex", "smooth", "smooth", "frame", "ensemble", "adjoint"])
    precision = rng.choice(["fp64", "fp64", "fp64", "bulk", "df64", "dev"])
    I = rng.choice([0.0, 1.0, 3.0])
    if kind in ("sod", "lax"):
        c = _case("", kind, precision, size(100, 8192), 1, size(20, 500), I)
    elif kind in ("sound", "vortex"):
        n = size(64, 4096)
        c = _case("", kind, precision, n, n, size(1, max(1, min(100, 10 * 4096 ** 2 // n ** 2))), I)
    elif kind in ("smooth", "frame"):
        nx, ny = size(33, 3000), size(33, 3000)
        c = _case("", kind, precision, nx, ny, size(1, max(1, min(100, 5 * 4096 ** 2 // (nx * ny)))), I, bc=rng.choice([0, 1]))
    elif kind == "ensemble":
        c = _case("", kind, precision, size(16, 1024), size(300, 4000), size(10, 100), I)
    else:
        n = size(32, 512)
        limiter = rng.choice([0, 1, 2])
        c = _case("", kind, "fp64", n, n, size(4, 40), I, every=rng.choice([5, 10, 20]), limiter=limiter)
    del c["name"]
    return c


# ------------------------------------------------------------------ inputs

def _periodic(w, rng, amp):
    """Two long waves in every field, of a few per cent or less: flow that is not aligned with the grid."""
    y, x = (np.arange(n) + 0.5 for n in (w.ny, w.nx))
    for k in FIELDS:
        a = np.array(getattr(w, k))
        for _ in range(2):
            p, q, ph = rng.integers(1, 4), rng.integers(1, 4), rng.uniform(0.0, 2.0 * np.pi, 2)
            a += rng.uniform(0.2, 1.0) * amp * np.outer(np.cos(2 * np.pi * q * y / w.ny + ph[1]), np.cos(2 * np.pi * p * x / w.nx + ph[0]))
        setattr(w, k, a)
    return w


def _tube(w, rng):
    """Left and right states a few per cent off the printed ones."""
    left = np.arange(w.nx) < w.nx // 2
    for k in ("rho", "T"):
        a, (l, r) = getattr(w, k), rng.uniform(0.95, 1.05, 2)
        setattr(w, k, a * np.where(left, l, r)[None, :])
    return w


def _workload(case, seed):
    rng = np.random.default_rng(seed)
    kind, nx, ny, I = case["kind"], case["nx"], case["ny"], case["I"]
    if kind in ("sod", "lax"):
        w = W.sod(nx=nx, I=I) if kind == "sod" else W.lax(nx=nx, I=I)
        w.dt = min(w.dt, 0.4 * w.dx / max(w.vg))
        return _tube(w, rng)
    if kind == "sound":
        w = W.sound(nx, I=I)
        w.dt = min(w.dt, 0.4 * w.dx / max(w.vg))
        return _periodic(w, rng, 1e-3)
    if kind == "vortex":
        return _periodic(W.taylor_green(nx, I=I, U0=rng.uniform(0.008, 0.012)), rng, 1e-3)
    if kind == "adjoint":
        return W.sound_modes(nx, seed=seed, I=I)
    dx, dy = 1.0 / nx, 1.0 / ny
    return W.random_smooth(nx, ny, seed=seed, I=I, dt=min(4e-4, 0.3 * min(dx, dy)), tau=1e-3, bc=(case["bc"], case["bc"]))


def _tubes(case, seed):
    """Lengths and I of the ensemble's draw of seed 0, left and right states of this seed's."""
    sizes, states = (W.ensemble_draw(case["nx"], seed=k, nx_lo=200, nx_hi=case["ny"]) for k in (0, seed))
    return [W.ensemble_tube({**s, "nx": z["nx"], "I": z["I"]}, steps=case["steps"]) for z, s in zip(sizes, states)]


def prepare(case, seed):
    kind, precision = case["kind"], PRECISIONS[case["precision"]]
    if kind == "ensemble":
        tubes = _tubes(case, seed)
        s = BatchSolver(tubes, precision=precision)
        s.init(tubes)
        s.set_tile(128, 4)
        return {"case": case, "solver": s, "tubes": tubes}
    w = _workload(case, seed)
    fields = [torch.from_numpy(np.ascontiguousarray(getattr(w, k))).cuda() for k in FIELDS]
    if kind == "adjoint":
        spec = {"nx": w.nx, "ny": w.ny, "dx": w.dx, "dy": w.dy, "dt": w.dt, "I": w.I, "vg": w.vg, "eg": w.eg, "limiter": case["limiter"]}
        target = torch.from_numpy(W.sound_modes(case["nx"], seed=seed + 1, I=case["I"]).rho).cuda()
        return {"case": case, "fields": fields, "tau": w.tau, "spec": spec, "target": target, "function": make_run_function()}
    s = Solver.from_workload(w, precision=precision)
    if kind == "frame":
        s.init(*fields)
        s.step(case["steps"])
    return {"case": case, "solver": s, "fields": fields}


# ------------------------------------------------------------------ one pass

def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "ensemble":
        s = state["solver"]
        s.init(state["tubes"])
        s.step(case["steps"])
        return dict(zip(FIELDS, s.macros()))
    if kind == "adjoint":
        leaves = [a.detach().requires_grad_(True) for a in state["fields"]]
        tau = torch.tensor(state["tau"], dtype=torch.float64, requires_grad=True)
        out = state["function"].apply(*leaves, tau, state["spec"], case["steps"], case["every"])
        loss = ((out[0] - state["target"]) ** 2).sum()
        loss.backward()
        res = {"loss": loss.detach(), "tau": tau.grad}
        res.update({k: v.detach() for k, v in zip(FIELDS, out)})
        res.update({"d_" + k: v.grad for k, v in zip(FIELDS, leaves)})
        return res
    s = state["solver"]
    if kind == "frame":
        res = dict(zip(FIELDS, s.macros()))
        res.update({"tne": s.tne(), "sums": s.conserved_sums()})
        return res
    s.init(*state["fields"])
    s.step(case["steps"])
    res = dict(zip(FIELDS, s.macros()))
    if case["steps"] > 1:
        res["f"] = s.state()      # the checkpoint of the run
    return res


# Floating-point operations of one cell in one step (two Runge-Kutta stages), a fused multiply-add as two.
_STEP_FLOPS = 766


def work(case):
    kind, steps = case["kind"], case["steps"]
    store = 8 if case["precision"] == "fp64" else 4
    if kind == "ensemble":
        cells = case["nx"] * (200 + case["ny"]) // 2
    else:
        cells = case["nx"] * case["ny"]
    if kind == "frame":      # the state read once; fields and Delta* written
        return {"bytes": cells * (16 * store + 8 * 16), "flops": cells * 450}
    io = cells * 8 * 8       # fields in and out
    if kind == "adjoint":
        # the run forward, and each step's transposed stages with their forward values; states that do
        # not fit on the chip are read and written once per step
        return {"bytes": io + cells * (5 * 8 + steps * 3 * 16 * store), "flops": cells * steps * _STEP_FLOPS * 3}
    if steps > 1:
        io += cells * 16 * 8 if kind != "ensemble" else 0
    # a state beyond the cache is read and written once per step
    through = steps * 2 * 16 * store * cells if 16 * store * cells > 100e6 and kind != "ensemble" else 0
    return {"bytes": io + through, "flops": cells * steps * _STEP_FLOPS}


# ------------------------------------------------------------------ the same in plain 64-bit torch

class _Model:
    """The method written out with torch operations: equilibrium from the inverse of the 16 moment
    rows at rest, minmod transport by index gathers, two-stage Runge-Kutta."""

    def __init__(self, vg, eg, I, tau, dt, lx, ly, xi, yi, dev):
        axis, diag = [(1, 0), (0, 1), (-1, 0), (0, -1)], [(1, 1), (-1, 1), (-1, -1), (1, -1)]
        self.dirs = [d for g in range(4) for d in (diag if g & 1 else axis)]
        vx = np.array([vg[i // 4] * d[0] for i, d in enumerate(self.dirs)])
        vy = np.array([vg[i // 4] * d[1] for i, d in enumerate(self.dirs)])
        w = vx ** 2 + vy ** 2 + np.repeat(np.array(eg), 4) ** 2
        rows = [vx ** 0, vx, vy, w, vx * vx, vx * vy, vy * vy, w * vx, w * vy, vx ** 3, vx * vx * vy, vx * vy * vy, vy ** 3,
                w * vx * vx, w * vx * vy, w * vy * vy]
        to = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64, device=dev)
        self.vx, self.vy, self.w, self.rows = to(vx), to(vy), to(w), to(np.stack(rows))
        self.inverse = to(np.linalg.inv(np.stack(rows)))
        self.I, self.K, self.tau, self.dt = I, 2.0 + I, tau, dt
        self.speed, self.lx, self.ly = [float(vg[i // 4]) for i in range(16)], lx, ly
        self.xi, self.yi = xi, yi     # {-2, -1, 1, 2} -> neighbour index along x, y
        self.freeze = 0

    def equilibrium(self, rho, u, v, T):
        x2, y2, I, K = u * u, v * v, self.I, self.K
        c, s = x2 + y2, u * v
        raw = [rho / rho, u, v, K * T + c, x2 + T, s, y2 + T, u * ((K + 2) * T + c), v * ((K + 2) * T + c), u * (x2 + 3 * T),
               v * (x2 + T), u * (y2 + T), v * (y2 + 3 * T),
               x2 * c + T * ((K + 5) * x2 + y2) + (K + 2) * T * T, s * (c + (K + 4) * T), y2 * c + T * ((K + 5) * y2 + x2) + (K + 2) * T * T]
        return torch.einsum("ik,k...->i...", self.inverse, torch.stack([rho * m for m in raw]))

    def fields(self, f):
        rho = f.sum(0)
        u, v = (torch.einsum("i,i...->...", a, f) / rho for a in (self.vx, self.vy))
        return rho, u, v, (torch.einsum("i,i...->...", self.w, f) / rho - u * u - v * v) / self.K

    def limited(self, X, Y):
        keep = ((X > 0) & (Y > 0)) | ((X < 0) & (Y < 0))
        small = X.detach().abs() <= Y.detach().abs()
        if self.freeze == 2:
            X, Y = X.detach(), Y.detach()
        if self.freeze == 1:   # the ratio of the result to the upwind difference is held
            n = torch.where(keep, torch.where(small, X, Y), torch.zeros_like(X)).detach()
            return Y * torch.where(Y == 0, torch.zeros_like(Y), n / Y).detach()
        return torch.where(keep, torch.where(small, X, Y), torch.zeros_like(X))

    def slope(self, p, s, at, dim):
        """Upwind-ordered (H(j + 1/2) - H(j - 1/2)) / |v| of one plane."""
        u2, u1, d1 = (p.index_select(dim, at[k * s]) for k in (-2, -1, 1))
        a = p - u1
        return a + 0.5 * (self.limited(d1 - p, a) - self.limited(a, u1 - u2))

    def rate(self, f):
        L = (self.equilibrium(*self.fields(f)) - f) / self.tau
        out = []
        for i, (sx, sy) in enumerate(self.dirs):
            r = L[i]
            if sx:
                r = r - self.speed[i] * self.lx * self.slope(f[i], sx, self.xi, -1)
            if sy and self.yi is not None:
                r = r - self.speed[i] * self.ly * self.slope(f[i], sy, self.yi, -2)
            out.append(r)
        return torch.stack(out)

    def step(self, f):
        g = f + self.dt * self.rate(f)
        return 0.5 * (f + g + self.dt * self.rate(g))

    def tne(self, f):
        rho, u, v, T = self.fields(f)
        d = f - self.equilibrium(rho, u, v, T)
        sh = (16,) + (1,) * (f.dim() - 1)
        cx, cy, eta2 = self.vx.view(sh) - u, self.vy.view(sh) - v, (self.w - self.vx ** 2 - self.vy ** 2).view(sh)
        w = cx * cx + cy * cy + eta2
        return torch.stack([(d * r).sum(0) for r in (cx * cx, cx * cy, cy * cy, w * cx, w * cy, cx ** 3, cx * cx * cy, cx * cy * cy, cy ** 3,
                                                     w * cx * cx, w * cx * cy, w * cy * cy)])

    def sums(self, f):
        t = f.sum((-2, -1))
        return torch.stack([t.sum(), (self.vx * t).sum(), (self.vy * t).sum(), (self.w * t).sum()])


def _neighbours(n, bc, dev):
    j = torch.arange(n, device=dev)
    return {k: (j + k) % n if bc == 0 else (j + k).clamp(0, n - 1) for k in (-2, -1, 1, 2)}


def _advance(model, f, steps):
    for _ in range(steps):
        f = model.step(f)
    return f


def _exact_ensemble(case, seed, dev):
    """The tubes end to end, one call per value of I, every cell with its own tube's ends."""
    tubes = _tubes(case, seed)
    res = {k: np.zeros(sum(w.nx for w in tubes)) for k in FIELDS}
    start = np.concatenate([[0], np.cumsum([w.nx for w in tubes])])
    for I in sorted({w.I for w in tubes}):
        ids = [t for t, w in enumerate(tubes) if w.I == I]
        n = np.array([tubes[t].nx for t in ids])
        lo = np.repeat(np.concatenate([[0], np.cumsum(n)[:-1]]), n)
        hi, j = lo + np.repeat(n, n) - 1, np.arange(n.sum())
        xi = {k: torch.from_numpy(np.clip(j + k, lo, hi)).to(dev) for k in (-2, -1, 1, 2)}
        w0 = tubes[ids[0]]
        lx = torch.from_numpy(np.repeat([1.0 / tubes[t].dx for t in ids], n)).to(dev)
        m = _Model(w0.vg, w0.eg, I, w0.tau, w0.dt, lx, 0.0, xi, None, dev)
        a = [torch.from_numpy(np.concatenate([getattr(tubes[t], k) for t in ids], axis=1)).to(dev) for k in FIELDS]
        out = m.fields(_advance(m, m.equilibrium(*a), case["steps"]))
        at = np.concatenate([np.arange(start[t], start[t + 1]) for t in ids])
        for k, v in zip(FIELDS, out):
            res[k][at] = v.cpu().numpy().reshape(-1)
    res["uy"] = None      # zero but for rounding
    return res


def exact(case, seed):
    kind, steps = case["kind"], case["steps"]
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if kind == "ensemble":
        return _exact_ensemble(case, seed, dev)
    w = _workload(case, seed)
    m = _Model(w.vg, w.eg, w.I, w.tau, w.dt, 1.0 / w.dx, 1.0 / w.dy, _neighbours(w.nx, w.bc_x, dev),
               _neighbours(w.ny, w.bc_y, dev) if w.ny > 1 else None, dev)
    a = [torch.from_numpy(np.ascontiguousarray(getattr(w, k))).to(dev) for k in FIELDS]
    if kind == "adjoint":
        m.freeze = case["limiter"]
        leaves = a + [torch.tensor(w.tau, dtype=torch.float64, device=dev)]
        for v in leaves:
            v.requires_grad_(True)
        m.tau = leaves[4]
        f = m.equilibrium(*leaves[:4])
        for _ in range(steps):
            f = torch.utils.checkpoint.checkpoint(m.step, f, use_reentrant=False)
        out = m.fields(f)
        target = torch.from_numpy(W.sound_modes(case["nx"], seed=seed + 1, I=case["I"]).rho).to(dev)
        loss = ((out[0] - target) ** 2).sum()
        loss.backward()
        res = {"loss": loss.detach(), "tau": leaves[4].grad}
        res.update({k: v.detach() for k, v in zip(FIELDS, out)})
        res.update({"d_" + k: v.grad for k, v in zip(FIELDS, leaves)})
        return res
    f = _advance(m, m.equilibrium(*a), steps)
    res = dict(zip(FIELDS, m.fields(f)))
    if kind == "frame":
        res.update({"tne": m.tne(f), "sums": m.sums(f)})
    elif steps > 1:
        res["f"] = f
    if w.ny == 1:
        res["uy"] = None      # zero but for rounding
    return res
