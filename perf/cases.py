"""Performance cases of the SPH pipeline: the calls a simulation program makes.

``listed()`` gives the fixed cases, ``draw(rng)`` more of the same ranges;
``prepare`` builds what a program holds before the call (a particle state on
the device and the library context), ``run`` makes one pass through the public
entry points, ``work`` counts the bytes and operations no implementation can
avoid, and ``exact`` evaluates the same equations in plain FP64 torch.

The setups are those of the tests and the benchmark: the periodic jittered
box, the Kelvin-Helmholtz shear layer, the rotating square patch, the ensemble
of jittered boxes and the uniform self-gravitating sphere.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2005_02656_gb300 import Ensemble, HostStepper, Params, Rollout, SphSim, rollout

DEV = "cuda:0"
STATE = ("x", "y", "z", "vx", "vy", "vz", "vxh", "vyh", "vzh", "h", "m", "u", "du_prev")
OUT = ("rho", "p", "c", "ax", "ay", "az", "du", "iad")
GAMMA, COURANT, DT_GROWTH, NG, SINC_N = 5.0 / 3.0, 0.2, 1.1, 100, 6
EPS = 1e-3                                  # gravitational softening of the sphere


def listed():
    # FP32-mixed runs that advance the state hold h fixed (ng=0, as the square-patch run does): with
    # the adaptation on, a neighbour count that flips on the last bit of a position moves h by 0.2%,
    # and outputs of two correct builds could no longer be compared
    return [
        # one full step of the 8,000-particle box: the smallest run people debug, convergence-test
        # and sweep parameters with, in both precisions; launches and latency count
        dict(name="step-box20-fp64", kind="step", setup="box", size=20, precision="fp64"),
        dict(name="step-box20-fp32", kind="step", setup="box", size=20, precision="fp32_mixed",
             ng=0),
        # an ordinary mid-size production step with a ragged particle count (250,047)
        dict(name="step-box63-fp32", kind="step", setup="box", size=63, precision="fp32_mixed",
             ng=0),
        # the headline: the 8.4M-particle shear layer, FP32-mixed
        dict(name="step-kh224-fp32", kind="step", setup="kh", size=224, precision="fp32_mixed",
             ng=0),
        # the same shear layer at 1/8 scale (1,067,054 particles), every operation in FP64
        dict(name="step-kh112-fp64", kind="step", setup="kh", size=112, precision="fp64"),
        # the rotating square patch (10^6 particles, open axes), driven stage by stage by a program
        # with its own integrator
        dict(name="stages-patch100-fp64", kind="stages", setup="patch", size=100, precision="fp64"),
        # the same stage calls with the grad-h terms switched on, 103,823 particles
        dict(name="stages-box47-gradh-fp32", kind="stages", setup="box", size=47,
             precision="fp32_mixed", gradh=1),
        # 256 uneven boxes (8^3 to 48^3) advanced together: a parameter study
        dict(name="ensemble-256", kind="ensemble", boxes=256, steps=4, precision="fp32_mixed",
             ng=0),
        # self-gravity of the uniform sphere: 998k particles FP32-mixed, 137k in FP64
        dict(name="gravity-sphere124-fp32", kind="gravity", setup="sphere", size=124, theta=0.5,
             precision="fp32_mixed"),
        dict(name="gravity-sphere64-fp64", kind="gravity", setup="sphere", size=64, theta=0.5,
             precision="fp64"),
        # forward and backward of a differentiable 20-step rollout with checkpoints every 5 steps
        dict(name="rollout-box40", kind="rollout", setup="box", size=40, steps=20, every=5,
             precision="fp64"),
        # a program whose state lives in pinned host memory, stepping a small box
        dict(name="host-box32-fp64", kind="host", setup="box", size=32, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "stages", "stages", "ensemble", "gravity",
                       "rollout", "host"])
    prec = rng.choice(["fp64", "fp32_mixed"])
    if kind in ("step", "stages"):
        # a step advances the state, so the patch (whose free surface fails after some tens of
        # steps) appears in the stage calls only
        setup = rng.choice(["box", "kh"] if kind == "step" else ["box", "kh", "patch"])
        if setup == "kh":
            size = 4 * _log_int(rng, 8, 24 if prec == "fp64" else 50)
        else:
            size = _log_int(rng, 12, 96 if prec == "fp64" else 150)
        case = dict(kind=kind, setup=setup, size=size, precision=prec)
        if kind == "step" and prec == "fp32_mixed":
            case["ng"] = 0
        option = rng.choice(["plain", "plain", "gradh", "table", "lists"])
        if option == "gradh":
            case["gradh"] = 1
        elif option == "table":
            case["kernel_mode"] = "table"
        elif option == "lists" and prec == "fp32_mixed":
            case["pair_mode"] = "lists"
        return case
    if kind == "ensemble":
        return dict(kind=kind, boxes=_log_int(rng, 8, 256), steps=rng.randint(1, 4),
                    precision="fp32_mixed", ng=0)
    if kind == "gravity":
        return dict(kind=kind, setup="sphere", size=_log_int(rng, 16, 72 if prec == "fp64" else 124),
                    theta=round(rng.uniform(0.4, 0.8), 2), precision=prec)
    if kind == "rollout":
        steps = rng.randint(2, 20)
        return dict(kind=kind, setup="box", size=_log_int(rng, 10, 40), steps=steps,
                    every=rng.randint(1, steps), precision="fp64")
    return dict(kind="host", setup="box", size=_log_int(rng, 12, 64), precision="fp64")


# --- inputs -----------------------------------------------------------------

def _lattice(nx, ny, nz, lo, dx):
    ax = [(torch.arange(k, dtype=torch.float64, device=DEV) + 0.5) * dx + o
          for k, o in zip((nx, ny, nz), lo)]
    z, y, x = torch.meshgrid(ax[2], ax[1], ax[0], indexing="ij")
    return [x.reshape(-1), y.reshape(-1), z.reshape(-1)]


def _h(dx):
    return dx * (3.0 * NG / (4.0 * math.pi)) ** (1.0 / 3.0) / 2.0


def _state(setup, size, seed):
    """A seeded particle state as device tensors, with the box, in random particle order."""
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)

    def uniform(n, a):
        return (2.0 * torch.rand(n, dtype=torch.float64, device=DEV, generator=g) - 1.0) * a

    lo, hi, periodic = (0.0, 0.0, 0.0), (1.0, 1.0, 1.0), (1, 1, 1)
    if setup == "kh":
        ni = 2 * int(round(size * 2.0 ** (1.0 / 3.0) / 2.0))
        do, di = 1.0 / size, 1.0 / ni
        parts = [_lattice(size, size // 4, size // 2, (0.0, y0, 0.0), do) for y0 in (0.0, 0.75)]
        parts.append(_lattice(ni, ni // 2, ni // 2, (0.0, 0.25, 0.0), di))
        x, y, z = (torch.cat(c) for c in zip(*parts))
        n, n_out = x.numel(), 2 * parts[0][0].numel()
        inner = torch.arange(n, device=DEV) >= n_out
        phase = float(uniform(1, math.pi))

        def either(a, b):
            return torch.where(inner, torch.full_like(x, a), torch.full_like(x, b))

        v = [either(0.5, -0.5), 0.01 * torch.sin(4.0 * math.pi * x + phase), torch.zeros_like(x)]
        # a run under way: the lattices have lost their exact symmetry
        x, y, z = (c + uniform(n, 0.05) * either(di, do) for c in (x, y, z))
        h, m = either(_h(di), _h(do)), either(0.5 / (n - n_out), 0.25 / n_out)
        u = either(2.5 / ((GAMMA - 1.0) * 2.0), 2.5 / (GAMMA - 1.0))
        hi = (1.0, 1.0, 0.5)
    elif setup == "patch":
        lo, hi, periodic = (-0.5,) * 3, (0.5,) * 3, (0, 0, 1)
        x, y, z = _lattice(size, size, size, lo, 1.0 / size)
        n = x.numel()
        x, y, z = (c + uniform(n, 0.05 / size) for c in (x, y, z))
        v = [5.0 * y, -5.0 * x, torch.zeros_like(x)]
        h, m, u = (torch.full_like(x, a) for a in (_h(1.0 / size), 1.0 / n, 1.0))
    else:
        sphere = setup == "sphere"
        dx = (2.0 if sphere else 1.0) / size
        lo = (-1.0,) * 3 if sphere else lo
        x, y, z = _lattice(size, size, size, lo, dx)
        if sphere:
            periodic = (0, 0, 0)
            keep = x * x + y * y + z * z < 1.0
            x, y, z = x[keep], y[keep], z[keep]
        n = x.numel()
        x, y, z = (c + uniform(n, 0.1 * dx) for c in (x, y, z))
        sigma = 0.0 if sphere else 0.01
        v = [sigma * torch.randn(n, dtype=torch.float64, device=DEV, generator=g) for _ in range(3)]
        h, m, u = (torch.full_like(x, a) for a in (_h(dx), 1.0 / n, 1.0))
    perm = torch.randperm(n, device=DEV, generator=g)
    s = dict(zip(STATE, (x, y, z, *v, *v, h, m, u, torch.zeros_like(x))))
    s = {k: a[perm].contiguous() for k, a in s.items()}
    s["id"] = perm.to(torch.int64)
    return s, dict(lo=lo, hi=hi, periodic=periodic)


def _host(s, box):
    return {**{k: a.cpu().numpy() for k, a in s.items()}, **box}


def _options(case):
    return {k: case[k] for k in ("gradh", "kernel_mode", "pair_mode") if k in case}


def _params(case, box):
    return Params(box_lo=box["lo"], box_hi=box["hi"], periodic=box["periodic"],
                  precision=case["precision"], ng_target=case.get("ng", NG), **_options(case))


def _boxes(case, seed):
    """(side, alpha) per box: sides log-uniform in [8, 48] (the study's own, the same for every
    seed), alpha uniform in [0.5, 1.5]."""
    sides = np.random.default_rng(case["boxes"]).uniform(math.log(8), math.log(48), case["boxes"])
    alpha = np.random.default_rng(seed).uniform(0.5, 1.5, case["boxes"])
    return list(zip(np.rint(np.exp(sides)).astype(int).tolist(), alpha.tolist()))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "ensemble":
        boxes = []
        for k, (side, alpha) in enumerate(_boxes(case, seed)):
            boxes.append((_host(*_state("box", side, seed * 1000 + k)), alpha))
        sim = Ensemble(boxes, Params(precision=case["precision"], ng_target=case["ng"]))
        sim.set_config(find_window=128)     # what the autotuner settles on for such boxes
        return dict(case=case, sim=sim, keys=STATE + OUT, snap=_snapshot(sim.t, STATE + OUT))
    s, box = _state(case["setup"], case["size"], seed)
    if kind == "rollout":
        n = s["x"].numel()
        ro = Rollout(n, case["steps"], case["every"], _params(case, box))
        x0 = torch.stack([s["x"], s["y"], s["z"]], 1).requires_grad_()
        v0 = torch.stack([s["vx"], s["vy"], s["vz"]], 1).requires_grad_()
        alpha = torch.tensor(1.0, dtype=torch.float64, device=DEV, requires_grad=True)
        return dict(case=case, ro=ro, x0=x0, v0=v0, u0=s["u"].requires_grad_(), alpha=alpha,
                    h=s["h"], m=s["m"])
    if kind == "host":
        return dict(case=case, sim=HostStepper(_host(s, box), _params(case, box)))
    sim = SphSim(_host(s, box), _params(case, box))
    keys = STATE + OUT + (("omega",) if case.get("gradh") else ())
    snap = _snapshot(sim.t, keys) if case["precision"] == "fp32_mixed" and kind != "gravity" else None
    return dict(case=case, sim=sim, keys=keys, snap=snap)


def _snapshot(t, keys):
    """Single-precision buffers of an FP32-mixed run's fields, as kept for output."""
    return {k: torch.empty(t[k].shape, dtype=torch.float32, device=DEV) for k in keys}


# --- one pass ---------------------------------------------------------------

def _fields(state):
    """What a program reads after the call: the state and the outputs; an FP32-mixed run's fields
    go to its single-precision snapshot (the pair sums carry no more than that)."""
    sim, snap = state["sim"], state["snap"]
    if snap is None:
        out = {k: sim.t[k] for k in state["keys"]}
    else:
        torch._foreach_copy_(list(snap.values()), [sim.t[k] for k in snap])
        out = dict(snap)
    out["id"] = sim.t["id"]
    return out


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "rollout":
        x, v, u, rho = rollout(state["x0"], state["v0"], state["u0"], state["alpha"], state["ro"],
                               state["h"], state["m"])
        loss = ((rho - 1.0) ** 2).sum() + 0.5 * (state["m"][:, None] * v * v).sum()
        grads = torch.autograd.grad(loss, (state["x0"], state["v0"], state["u0"], state["alpha"]))
        return [x, v, u, rho, *grads]
    sim = state["sim"]
    if kind == "host":
        sim.step()
        return {**{k: sim.h[k] for k in STATE}, "id": sim.h["id"], "dt": sim.dt}
    if kind == "gravity":
        g, counts = sim.gravity(1.0, EPS, case["theta"])
        return {"g": g.float() if case["precision"] == "fp32_mixed" else g, "counts": counts,
                "id": sim.t["id"]}
    if kind == "stages":
        sim.find_neighbors()
        sim.density()
        sim.iad()
        sim.momentum_energy()
        return _fields(state)
    sim.step(case["steps"]) if kind == "ensemble" else sim.step()
    out = _fields(state)
    out["dt"] = sim.dt if state["snap"] is None else sim.dt.float()
    return out


# --- work -------------------------------------------------------------------

def _count(case):
    if case["kind"] == "ensemble":          # mean of side^3, side log-uniform in [8, 48]
        return case["boxes"] * (48 ** 3 - 8 ** 3) / (3.0 * math.log(6.0))
    k = case["size"]
    if case["setup"] == "kh":
        ni = 2 * int(round(k * 2.0 ** (1.0 / 3.0) / 2.0))
        return 2 * k * (k // 4) * (k // 2) + ni * (ni // 2) ** 2
    return k ** 3 * (math.pi / 6.0 if case["setup"] == "sphere" else 1.0)


def work(case):
    """Bytes: the state read and the state and outputs written, once.  Operations: those of the
    equations per neighbour pair (100 per particle; 14 for the distance test, and density, IAD and
    momentum), per tree interaction, and for the gradient twice the forward's on top of it."""
    n, kind, fp64 = _count(case), case["kind"], case["precision"] == "fp64"
    pair = 14 + 43 + 19 + 131 if fp64 else 14 + 37 + 57 + 140
    if kind == "gravity":
        # about 700 node and 800 particle terms per target at theta = 0.5 for 10^6 particles
        terms = (0.5 / case["theta"]) ** 2 * max(0.1, 1.0 + 0.15 * math.log(n / 1e6))
        return {"bytes": n * (5 * 8 + 3 * (8 if fp64 else 4)), "flops": n * terms * (700 * 65 + 800 * 21)}
    if kind == "rollout":
        steps = case["steps"]
        return {"bytes": n * 8 * (13 * steps + 2 * 13), "flops": n * NG * pair * 3.0 * steps}
    steps = case.get("steps", 1)
    written = 14 + 13 if kind != "host" else 14
    return {"bytes": n * 8 * (14 + written), "flops": float(n * NG * pair * steps)}


# --- the same equations in plain FP64 -----------------------------------------

def _norm():
    """B_n of the sinc kernel: 4 pi B int_0^2 S(v)^n v^2 dv = 1 (Gauss-Legendre)."""
    q, w = np.polynomial.legendre.leggauss(100)
    v = q + 1.0
    return 1.0 / (4.0 * math.pi * math.fsum(w * np.sinc(v / 2.0) ** SINC_N * v * v))


def _S6(v, table):
    if table is None:
        return torch.sinc(0.5 * v) ** SINC_N
    q = v * (0.5 * (table.numel() - 1))
    i = q.to(torch.int64).clamp_(max=table.numel() - 2)
    return table[i] + (table[i + 1] - table[i]) * (q - i)


def _spread(v):
    out = torch.zeros_like(v)
    for b in range(8):
        out |= ((v >> b) & 1) << (3 * b)
    return out


class _Grid:
    """Cells of side >= 2 h_max in Morton order, at most 256 per axis."""

    def __init__(self, s, box):
        self.pos = [s[k] for k in "xyz"]
        self.h, self.box = s["h"], box
        hmax = float(self.h.max())
        self.lo, self.nc, self.inv = [], [], []
        for k, p in enumerate(self.pos):
            lo, hi = (box["lo"][k], box["hi"][k]) if box["periodic"][k] else (float(p.min()), float(p.max()))
            nc = min(max(int((hi - lo) / (2.0 * hmax * (1.0 + 1e-9))), 1), 256)
            self.lo.append(lo)
            self.nc.append(nc)
            self.inv.append(1.0 / ((hi - lo) / nc))
        self.cell = [((p - lo) * inv).floor().to(torch.int64).clamp_(0, nc - 1)
                     for p, lo, inv, nc in zip(self.pos, self.lo, self.inv, self.nc)]

    def order(self):
        """Morton order of the cells, the previous order within a cell."""
        code = _spread(self.cell[0]) | (_spread(self.cell[1]) << 1) | (_spread(self.cell[2]) << 2)
        return torch.argsort(code, stable=True)

    def sep(self, a, b, k):
        d = self.pos[k][b] - self.pos[k][a]
        if self.box["periodic"][k]:
            L = self.box["hi"][k] - self.box["lo"][k]
            d = torch.where(d > 0.5 * L, d - L, torch.where(d < -0.5 * L, d + L, d))
        return d

    @torch.no_grad()
    def pairs(self, chunk=200_000):
        """(a, b) index tensors of the pairs with r_ab < 2 h_a, b != a, a ascending, in chunks."""
        nx, ny, nz = self.nc
        flat = self.cell[0] + nx * (self.cell[1] + ny * self.cell[2])
        by_cell = torch.argsort(flat, stable=True)
        count = torch.bincount(flat, minlength=nx * ny * nz)
        start = torch.cumsum(count, 0) - count
        offs = [[0] if c == 1 else [0, 1] if c == 2 and per else [-1, 0, 1]
                for c, per in zip(self.nc, self.box["periodic"])]
        n, found = self.h.numel(), []
        for t0 in range(0, n, chunk):
            t = torch.arange(t0, min(n, t0 + chunk), device=DEV)
            aa, bb = [], []
            for oz in offs[2]:
                for oy in offs[1]:
                    for ox in offs[0]:
                        ok, q = torch.ones_like(t, dtype=torch.bool), []
                        for c, o, nc, per in zip(self.cell, (ox, oy, oz), self.nc, self.box["periodic"]):
                            v = c[t] + o
                            if not per:
                                ok &= (v >= 0) & (v < nc)
                            q.append(v % nc)
                        f = q[0] + nx * (q[1] + ny * q[2])
                        cnt = torch.where(ok, count[f], torch.zeros_like(f))
                        a = torch.repeat_interleave(t, cnt)
                        first = torch.repeat_interleave(start[f] - (torch.cumsum(cnt, 0) - cnt), cnt)
                        b = by_cell[first + torch.arange(a.numel(), device=DEV)]
                        dx, dy, dz = (self.sep(a, b, k) for k in range(3))
                        r2, lim = (dx * dx + dy * dy) + dz * dz, 2.0 * self.h[a]
                        hit = (r2 < lim * lim) & (a != b)
                        aa.append(a[hit])
                        bb.append(b[hit])
            found.append((torch.cat(aa), torch.cat(bb)))
        return found


def _add(n, a, v):
    return torch.zeros(n, dtype=torch.float64, device=DEV).index_add(0, a, v)


def _inverse(t):
    """Inverse of the symmetric matrices xx xy xz yy yz zz (a list of six tensors)."""
    t00, t01, t02, t11, t12, t22 = t
    c = [t11 * t22 - t12 * t12, t02 * t12 - t01 * t22, t01 * t12 - t02 * t11,
         t00 * t22 - t02 * t02, t01 * t02 - t00 * t12, t00 * t11 - t01 * t01]
    det = t00 * c[0] + t01 * c[1] + t02 * c[2]
    return [q / det for q in c]


def _mul(c, d):
    return [c[0] * d[0] + c[1] * d[1] + c[2] * d[2], c[1] * d[0] + c[3] * d[1] + c[4] * d[2],
            c[2] * d[0] + c[4] * d[1] + c[5] * d[2]]


def _density(s, grid, pairs, opts):
    n, h, m = s["x"].numel(), s["h"], s["m"]
    Bn, table = _norm(), opts.get("table")
    rho, dsum = m * (Bn / h ** 3), -3.0 * m * (Bn / h ** 4)
    for a, b in pairs:
        v = torch.sqrt(sum(grid.sep(a, b, k) ** 2 for k in range(3))) / h[a]
        S6 = _S6(v, table)
        rho = rho + _add(n, a, m[b] * (Bn / h[a] ** 3) * S6)
        if opts.get("gradh"):
            x = 0.5 * math.pi * v
            S = torch.sinc(0.5 * v)
            dW = Bn / h[a] ** 3 * SINC_N * S ** (SINC_N - 1) * (torch.cos(x) - S) / v
            dsum = dsum + _add(n, a, -m[b] * (3.0 * Bn / h[a] ** 3 * S6 + v * dW) / h[a])
    p = (GAMMA - 1.0) * rho * s["u"]
    omega = 1.0 + h / (3.0 * rho) * dsum if opts.get("gradh") else torch.ones_like(rho)
    return rho, p, torch.sqrt(GAMMA * p / rho), omega


def _forces(s, grid, pairs, opts, alpha=1.0):
    """Density, equation of state, IAD matrices, accelerations and du/dt."""
    n, h, m = s["x"].numel(), s["h"], s["m"]
    Bn, table = _norm(), opts.get("table")
    rho, p, c, omega = _density(s, grid, pairs, opts)
    vol, tau = m / rho, [0.0] * 6
    for a, b in pairs:
        d = [grid.sep(a, b, k) for k in range(3)]
        w = vol[b] * (Bn / h[a] ** 3) * _S6(torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2) / h[a], table)
        tau = [q + _add(n, a, w * d[i] * d[j])
               for q, (i, j) in zip(tau, ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2)))]
    C = _inverse(tau)
    X, vel = p / (omega * rho ** 2), [s[k] for k in ("vx", "vy", "vz")]
    acc = [0.0] * 4
    for a, b in pairs:
        d = [grid.sep(a, b, k) for k in range(3)]
        r = torch.sqrt(d[0] ** 2 + d[1] ** 2 + d[2] ** 2)
        Wa = Bn / h[a] ** 3 * _S6(r / h[a], table)
        vb = (r / h[b]).clamp(max=2.0)
        Wb = Bn / h[b] ** 3 * _S6(vb, table)
        Aa = [q * Wa for q in _mul([e[a] for e in C], d)]
        Ab = [q * Wb for q in _mul([e[b] for e in C], d)]
        vab = [q[a] - q[b] for q in vel]
        xv = -(d[0] * vab[0] + d[1] * vab[1] + d[2] * vab[2])
        w = xv / r
        Pi = torch.where(xv.detach() < 0.0, -0.5 * alpha * (c[a] + c[b] - 3.0 * w) * w, torch.zeros_like(w))
        Abar = [i / rho[a] + j / rho[b] for i, j in zip(Aa, Ab)]
        va, vbar = (sum(i * j for i, j in zip(vab, q)) for q in (Aa, Abar))
        terms = [-m[b] * (X[a] * i + X[b] * j) - 0.5 * m[b] * Pi * k for i, j, k in zip(Aa, Ab, Abar)]
        terms.append(m[b] * (X[a] * va + 0.25 * Pi * vbar))
        acc = [q + _add(n, a, t) for q, t in zip(acc, terms)]
    out = dict(rho=rho, p=p, c=c, ax=acc[0], ay=acc[1], az=acc[2], du=acc[3],
               iad=torch.stack(C, 1).reshape(-1))
    return {**out, "omega": omega} if opts.get("gradh") else out


def _sorted(s, box):
    o = _Grid(s, box).order()
    s = {k: v[o] for k, v in s.items()}
    return s, _Grid(s, box)


def _advance(s, box, opts, alpha, dt_prev, ng):
    """One step: the sorted new state, the outputs and the time step."""
    s, grid = _sorted(s, box)
    pairs = grid.pairs()
    nn = sum(torch.bincount(a, minlength=s["x"].numel()) for a, _ in pairs).clamp(min=1)
    out = _forces(s, grid, pairs, opts, alpha)
    dt = COURANT * float((s["h"].detach() / out["c"].detach()).min())
    dt = min(dt, DT_GROWTH * dt_prev) if dt_prev > 0.0 else dt
    new = dict(s)
    for k, ax in enumerate("xyz"):
        vh = s["v" + ax + "h"] + out["a" + ax] * (0.5 * (dt + dt_prev))
        x = s[ax] + dt * vh
        if box["periodic"][k]:
            lo, hi = box["lo"][k], box["hi"][k]
            x = torch.where(x >= hi, x - (hi - lo), torch.where(x < lo, x + (hi - lo), x))
        new[ax], new["v" + ax + "h"], new["v" + ax] = x, vh, vh + 0.5 * dt * out["a" + ax]
    q = dt / (2.0 * dt_prev) if dt_prev > 0.0 else 0.0
    new["u"] = s["u"] + dt * ((1.0 + q) * out["du"] - q * s["du_prev"])
    new["du_prev"] = out["du"]
    if ng > 0:
        new["h"] = s["h"] * 0.5 * (1.0 + (ng / nn.double()) ** (1.0 / 3.0))
    return new, out, dt


def _gravity(s, chunk=512):
    pos = torch.stack([s["x"], s["y"], s["z"]])
    g = []
    for t0 in range(0, pos.shape[1], chunk):
        d = pos[:, None, :] - pos[:, t0:t0 + chunk, None]
        w = s["m"] * torch.rsqrt((d * d).sum(0) + EPS * EPS) ** 3
        g.append((d * w).sum(-1))
    return torch.cat(g, 1).t()


def exact(case, seed):
    kind, opts = case["kind"], {"gradh": case.get("gradh", 0)}
    if case.get("kernel_mode") == "table":
        opts["table"] = torch.sinc(torch.linspace(0.0, 1.0, 20000, dtype=torch.float64, device=DEV)) ** SINC_N
    if kind == "ensemble":
        done = []
        for k, (side, alpha) in enumerate(_boxes(case, seed)):
            s, box = _state("box", side, seed * 1000 + k)
            dt = 0.0
            for _ in range(case["steps"]):
                s, out, dt = _advance(s, box, opts, alpha, dt, case.get("ng", NG))
            done.append({**s, **out, "dt": torch.tensor([dt], device=DEV, dtype=torch.float64)})
        return {k: torch.cat([d[k] for d in done]) for k in done[0]}
    s, box = _state(case["setup"], case["size"], seed)
    if kind == "gravity":
        if s["x"].numel() > 200_000:        # the direct sum takes too long
            return None
        s, _ = _sorted(s, box)
        return {"g": _gravity(s), "counts": None, "id": s["id"]}
    if kind == "rollout":
        return _exact_rollout(case, s, box, opts)
    if kind == "stages":
        s, grid = _sorted(s, box)
        return {**s, **_forces(s, grid, grid.pairs(), opts)}
    new, out, dt = _advance(s, box, opts, 1.0, 0.0, case.get("ng", NG))
    dt = torch.tensor([dt], dtype=torch.float64)
    return {**new, "dt": dt} if kind == "host" else {**new, **out, "dt": dt}


def _exact_rollout(case, s, box, opts):
    """Reverse-mode differentiation of the rollout with lists, h and dt held; None where the graph
    of all steps' pair sums would not fit."""
    if s["x"].numel() * (case["steps"] + 1) > 1_500_000:
        return None
    x0, v0 = (torch.stack([s[k + e] for e in "xyz"], 1).requires_grad_() for k in ("", "v"))
    u0, alpha = s["u"].requires_grad_(), torch.tensor(1.0, dtype=torch.float64, device=DEV, requires_grad=True)
    s = {**s, "u": u0, "id": torch.arange(u0.numel(), device=DEV)}
    for k, e in enumerate("xyz"):
        s[e], s["v" + e], s["v" + e + "h"] = x0[:, k], v0[:, k], v0[:, k]
    dt = 0.0
    for _ in range(case["steps"]):
        s, _, dt = _advance(s, box, opts, alpha, dt, case.get("ng", NG))
    s, grid = _sorted(s, box)
    rho = _density(s, grid, grid.pairs(), opts)[0]
    back = torch.argsort(s["id"])
    x, v = (torch.stack([s[k + e] for e in "xyz"], 1) for k in ("", "v"))
    loss = ((rho - 1.0) ** 2).sum() + 0.5 * (s["m"][:, None] * v * v).sum()
    grads = torch.autograd.grad(loss, (x0, v0, u0, alpha))
    return [x[back], v[back], s["u"][back], rho[back], *grads]
