"""The work that users of this framework have it do, as cases that can be
timed and checked: stepping tubes and two-dimensional shock problems in each
precision, the batched sweep, gradients through a run, the stability scan and
the read-out of a large state.

Every case goes through the public entry points (``lbm.Lattice``,
``lbm.Batch``, ``autodiff.run``, ``lbm.vn_scan``).  ``exact`` states the same
results in 64 bits with plain torch and numpy, written from the scheme's
formulas: nothing of the library's arithmetic is used there, only the problem
descriptions of ``workloads``.
"""
from __future__ import annotations

import math

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_0706_0405_gb300 import autodiff, lbm
from paper_0706_0405_gb300 import workloads as W

DEV = "cuda"
FP32_MODES = ("fp32_tdf", "fp32_cons", "fp32", "fp32_t64")
DIRS = lbm.DIRECTIONS
NK = 31  # wave numbers per direction, as in the paper's Figs. 2-7


def listed():
    return [
        # The plain method in the default precision on the smallest grid of the
        # repository, watched as it runs: totals every 20 steps.  Latency and
        # launches are all of it.
        {"name": "sod_400x4_fp64", "kind": "watch", "problem": "sod", "nx": 400, "precision": "fp64",
         "steps": 20, "frames": 10},
        # The 1000:1 tube in the headline mode: thousands of very short steps.
        {"name": "tube_2000x4_tdf", "kind": "run", "problem": "ratio1000", "nx": 2000,
         "precision": "fp32_tdf", "steps": 500},
        # The paper's own double Mach reflection grid, a small 2-D run with all
        # four boundary kinds and a moving top boundary.
        {"name": "dmr_400x100_tdf", "kind": "run", "problem": "dmr", "ny": 100, "precision": "fp32_tdf",
         "steps": 400},
        # Regular reflection (Fig. 11): sizes that no tile divides.
        {"name": "regref_900x300_cons", "kind": "run", "problem": "regref", "ny": 300,
         "precision": "fp32_cons", "steps": 200},
        # The quarter-size double Mach reflection of the accuracy runs, with the
        # temperature recovered in FP64.
        {"name": "dmr_1024x256_t64", "kind": "run", "problem": "dmr", "ny": 256, "precision": "fp32_t64",
         "steps": 100},
        # The same grid in FP64: the reference run that the FP32 modes are held to.
        {"name": "dmr_1024x256_fp64", "kind": "run", "problem": "dmr", "ny": 256, "precision": "fp64",
         "steps": 40},
        # The headline workload of bench.py: the large grid, larger than L2.
        {"name": "dmr_4096x1024_tdf", "kind": "run", "problem": "dmr", "ny": 1024,
         "precision": "fp32_tdf", "steps": 20},
        # Restart and read-out of a large state: the saved f goes in, moments,
        # FP64 totals and f come out.
        {"name": "readout_4096x1024_cons", "kind": "readout", "problem": "dmr", "ny": 1024,
         "precision": "fp32_cons"},
        # The batched sweep of 256 uneven Riemann tubes.
        {"name": "batch_256_tdf", "kind": "batch", "count": 256, "precision": "fp32_tdf", "steps": 500},
        # Gradient of a final-density misfit through the Mach-3 tube, forward and
        # backward with a checkpoint every 50 steps.
        {"name": "grad_2048x256_tdf", "kind": "grad", "nx": 2048, "ny": 256, "precision": "fp32_tdf",
         "steps": 100, "every": 50},
        # The same gradient on the reduced tube of the tests in the default
        # precision: short kernels, many launches and allocations.
        {"name": "grad_256x8_fp64", "kind": "grad", "nx": 256, "ny": 8, "precision": "fp64", "steps": 200,
         "every": 50},
        # Vetting the time step of the whole sweep: the left and right states of
        # its 256 tubes in four directions.
        {"name": "vn_256", "kind": "vn", "count": 256},
    ]


def draw(rng):
    """One more case: any kind, sizes spread over the logarithm of the range,
    any precision, at most the listed ones' work."""
    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "run", "watch", "readout", "batch", "grad", "vn"])
    prec = rng.choice(("fp64",) + FP32_MODES)
    # node updates of one pass: FP64 is slower on this part, so it gets fewer
    most = 10_000_000 if prec in ("fp64", "fp32_t64") else 80_000_000
    if kind in ("run", "watch", "readout"):
        problem = rng.choice(["sod", "ratio1000", "mach30", "dmr", "regref"])
        case = {"kind": kind, "problem": problem, "precision": prec}
        if problem in ("dmr", "regref"):
            big = 1024 if prec not in ("fp64", "fp32_t64") else 512
            case["ny"] = log_int(24, big if problem == "dmr" else big // 2)
            nodes = (4 if problem == "dmr" else 3) * case["ny"] ** 2
        else:
            case["nx"] = log_int(96, 4096)
            nodes = 4 * case["nx"]
        if kind != "readout":
            case["steps"] = max(2, min(log_int(5, 500), most // nodes))
        if kind == "watch":
            case["frames"] = rng.randint(2, 8)
            case["steps"] = max(1, min(case["steps"], most // nodes) // case["frames"])
        return case
    if kind == "batch":
        return {"kind": "batch", "count": log_int(4, 256), "precision": rng.choice(FP32_MODES),
                "steps": log_int(20, 400)}
    if kind == "grad":
        nx, ny = log_int(64, 1024), log_int(4, 128)
        return {"kind": "grad", "nx": nx, "ny": ny, "precision": prec,
                "steps": max(10, min(log_int(20, 200), most // (8 * nx * ny))), "every": rng.choice([8, 16, 50])}
    return {"kind": "vn", "count": log_int(8, 256)}


# ------------------------------------------------------------------ inputs

def _problem(case):
    name = case["problem"] if "problem" in case else "mach3"
    if name == "sod":
        nx = case["nx"]
        return W.riemann("sod", nx, 4, 1.0, (1.0, 0.0, 0.0, 1.0), (0.125, 0.0, 0.0, 0.1), 0.5, 3.0, 9.0, 5.0,
                         alpha=0.036)
    if name == "ratio1000":
        nx = case["nx"]
        return W.riemann("ratio1000", nx, 4, 0.0025 * nx, (1000.0, 0.0, 0.0, 1000.0), (1.0, 0.0, 0.0, 1.0),
                         0.00125 * nx, 3.0, 9.0, 5.0, alpha=0.05)
    if name == "mach30":
        return W.mach30_tube(case["nx"])
    if name == "dmr":
        return W.dmr_paper() if case["ny"] == 100 else W.dmr(case["ny"])
    if name == "regref":
        return W.regular_reflection(case["ny"])
    nx, ny = case["nx"], case["ny"]
    return W.riemann("mach3", nx, ny, 1.0, (1.4, 3.0, 0.0, 1.0), (1.4, 0.0, 0.0, 1.0), 0.5, 4.0, 10.0, 6.0,
                     alpha=0.05)


def _dtype(case):
    return torch.float64 if case["precision"] == "fp64" else torch.float32


def _fields(p, gen, dtype, sigma=1e-3):
    """The problem's initial (rho, ux, uy, T) with a Gaussian perturbation of
    sigma times the local rho and T, and times the flow speed for u."""
    base = [torch.as_tensor(a, device=DEV) for a in W.initial_fields(p)]
    speed = max(1.0, abs(p.setup.get("left", (0.0, 1.0))[1]))
    scale = (base[0], speed, speed, base[3])
    return [(b + sigma * s * torch.randn(b.shape, dtype=torch.float64, device=DEV, generator=gen)).to(dtype)
            for b, s in zip(base, scale)]


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _inputs(case, seed):
    """(problem(s), inputs) of a case: what its user has in hand."""
    kind = case["kind"]
    gen = _gen(seed)
    if kind == "vn":
        # the sweep's tubes, each at its left and right state, slightly moved
        rng = np.random.Generator(np.random.PCG64(seed))
        states = []
        for p in W.batch_riemann(case["count"]):
            for side in ("left", "right"):
                r, u, v, t = p.setup[side]
                m = 1.0 + 0.01 * rng.standard_normal(4)
                states.append((p, (r * m[0], u * m[1], 0.05 * m[2], t * m[3])))
        return None, states
    if kind == "batch":
        probs = W.batch_riemann(case["count"])
        return probs, [_fields(p, gen, torch.float32) for p in probs]
    p = _problem(case)
    dtype = _dtype(case)
    if kind == "grad":
        fields = _fields(p, gen, dtype, 0.01)
        target = _fields(p, gen, dtype, 0.01)[0]
        return p, (fields, target)
    fields = _fields(p, gen, dtype)
    if kind == "readout":
        # a state away from equilibrium, as a run leaves it
        f = _equilibrium(_Scheme(p), *[a.double() for a in fields])
        return p, (f * (1.0 + 1e-3 * torch.randn(f.shape, dtype=torch.float64, device=DEV, generator=gen))).to(dtype)
    return p, fields


def prepare(case, seed):
    kind = case["kind"]
    p, given = _inputs(case, seed)
    state = {"case": case, "kind": kind, "in": given}
    if kind == "vn":
        state["cases"] = [lbm.vn_case(q, s) for q, s in given]
    elif kind == "batch":
        b = lbm.Batch(p, case["precision"])
        ny, total = p[0].ny, sum(q.nx for q in p)
        # one flat output per quantity, each tube's ny x nx block after the other
        out = [torch.empty(ny * total, dtype=torch.float32, device=DEV) for _ in range(4)]
        views, at = [], 0
        for q in p:
            views.append([o[at:at + q.nx * ny] for o in out])
            at += q.nx * ny
        # per quantity, the tubes' arrays, as lbm_batch_init takes them
        state["in"] = [[g[q] for g in given] for q in range(4)]
        lbm.lbm_batch_init(b.handle, *state["in"])
        b.autotune()
        state.update(b=b, out=out, views=views)
    elif kind == "grad":
        state["p"] = p
        state["tau"] = torch.tensor(p.tau, dtype=_dtype(case), requires_grad=True)
        state["fields"] = [a.requires_grad_(True) for a in given[0]]
    else:
        state["lat"] = lbm.Lattice(p, case["precision"])
    return state


def run(state):
    case, kind = state["case"], state["kind"]
    if kind == "run":
        lat = state["lat"]
        return dict(zip(("rho", "ux", "uy", "T"), lat.init(*state["in"]).step(case["steps"]).moments()))
    if kind == "watch":
        lat = state["lat"].init(*state["in"])
        totals = []
        for _ in range(case["frames"]):
            totals.append(lat.step(case["steps"]).conservation())
        return {"totals": np.stack(totals), **dict(zip(("rho", "ux", "uy", "T"), lat.moments()))}
    if kind == "readout":
        lat = state["lat"].set_f(state["in"], 7)
        out = dict(zip(("rho", "ux", "uy", "T"), lat.moments()))
        return {**out, "totals": lat.conservation(), "f": lat.get_f()}
    if kind == "batch":
        b = state["b"]
        lbm.lbm_batch_init(b.handle, *state["in"])
        b.step(case["steps"])
        for k, views in enumerate(state["views"]):
            lbm.lbm_moments(lbm.lbm_batch_problem(b.handle, k), *views)
        b.sync()
        return dict(zip(("rho", "ux", "uy", "T"), state["out"]))
    if kind == "grad":
        fields, target = state["fields"], state["in"][1]
        out = autodiff.run(state["p"], *fields, state["tau"], case["steps"], every=case["every"],
                           precision=case["precision"])
        loss = 0.5 * torch.sum((out[0] - target) ** 2)
        grads = torch.autograd.grad(loss, [*fields, state["tau"]])
        return {"out": [a.detach() for a in out], "grads": list(grads)}
    radius, growth = lbm.vn_scan(state["cases"], DIRS, NK)
    return {"radius": radius, "growth": growth}


def work(case):
    """Bytes of the inputs and outputs; arithmetic of the plain method, about
    200 operations per node and step (moments 40, equilibrium 50, relaxation
    and five-point update 110), of its transpose about 330, and of one 9 x 9
    complex eigenvalue problem about 40 n^3."""
    kind = case["kind"]
    if kind == "vn":
        m = 2 * case["count"] * len(DIRS) * NK
        return {"bytes": 8 * m + 400 * case["count"], "flops": 40 * 729 * m}
    if kind == "batch":
        nodes, size = sum(p.nodes for p in W.batch_riemann(case["count"])), 4
    else:
        nodes, size = _problem(case).nodes, 8 if case["precision"] == "fp64" else 4
    if kind == "readout":
        return {"bytes": (9 + 4 + 9) * size * nodes, "flops": 80 * nodes}
    steps = case["steps"] * case.get("frames", 1)
    if kind == "grad":
        return {"bytes": (5 + 4 + 4) * size * nodes, "flops": (2 * 200 + 330) * steps * nodes}
    return {"bytes": 8 * size * nodes, "flops": 200 * steps * nodes}


# ----------------------------------------------------- the scheme in 64 bits

SX = (0, -1, 0, 1, 0, -1, 1, 1, -1)
SY = (0, 0, -1, 0, 1, -1, -1, 1, 1)
MIRROR_X = [0, 3, 2, 1, 4, 6, 5, 8, 7]
MIRROR_Y = [0, 1, 4, 3, 2, 8, 7, 6, 5]


class _Scheme:
    """Constants of the D2V9 model and of the five-point update for one
    problem, or column by column for a list of problems (each constant then a
    row vector over the columns)."""

    def __init__(self, p, tau=None):
        many = isinstance(p, (list, tuple))
        if many:
            def col(fn):
                return torch.cat([torch.full((q.nx,), float(fn(q)), dtype=torch.float64) for q in p]).to(DEV)[None]
        else:
            def col(fn):
                return float(fn(p))
        self.c1, self.c2, self.eta = col(lambda q: q.c1), col(lambda q: q.c2), col(lambda q: q.eta0)
        self.b, dt, dx = col(lambda q: q.b), col(lambda q: q.dt), col(lambda q: q.dx)
        self.omega = dt / (col(lambda q: q.tau) if tau is None else tau)
        d = self.c2 / math.sqrt(2.0)
        mag = [0.0 * self.c1] + [self.c1] * 4 + [d] * 4
        self.vx = [s * m for s, m in zip(SX, mag)]
        self.vy = [s * m for s, m in zip(SY, mag)]
        beta = col(lambda q: q.beta)
        self.adv = []  # weights of (centre, east, west, north, south) without the relaxation
        for i in range(9):
            mu = col(lambda q: q.lam[i]) * dt / dx ** 2
            c, w = -4.0 * mu, []
            for v, up in ((self.vx[i] * dt / dx, SX[i] >= 0), (self.vy[i] * dt / dx, SY[i] >= 0)):
                if up:
                    plus, here, minus = beta, 1.0 - 2.0 * beta, -(1.0 - beta)
                else:
                    plus, here, minus = 1.0 - beta, -(1.0 - 2.0 * beta), -beta
                c = c - v * here
                w += [mu - v * plus, mu - v * minus]
            self.adv.append((c, *w))


def _moments(s, f):
    rho = f.sum(0)
    ux = sum(s.vx[i] * f[i] for i in range(1, 9)) / rho
    uy = sum(s.vy[i] * f[i] for i in range(1, 9)) / rho
    inner = sum(f[i] * ((s.vx[i] - ux) ** 2 + (s.vy[i] - uy) ** 2) for i in range(9)) + f[0] * s.eta ** 2
    return rho, ux, uy, inner / (s.b * rho)


def _equilibrium(s, rho, ux, uy, T):
    c1s, c2s, e = s.c1 ** 2, s.c2 ** 2, s.eta ** 2
    u2 = ux * ux + uy * uy
    out = [rho * (s.b - 2.0) * T / e]
    for i in range(1, 9):
        own, other = (c1s, c2s) if i <= 4 else (c2s, c1s)
        A = (-other + ((s.b - 2.0) * other / e + 2.0) * T + other / own * u2) / (4.0 * (own - other))
        B = (-other + (s.b + 2.0) * T + u2) / (2.0 * own * (own - other))
        vu = s.vx[i] * ux + s.vy[i] * uy
        out.append(rho * (A + B * vu + vu * vu / (2.0 * own ** 2)))
    return torch.stack(out)


def _part(side, along, t):
    """True where a side's cell at `along` lies below its split at time t."""
    return along < side.split0 + side.split_speed * t


def _neighbours(p, s, f, level):
    """East, west, north and south values of every node, ghost cells by the
    boundary rules at the level's time."""
    t = level * p.dt
    ny, nx = f.shape[1:]
    lens = {0: ny, 1: ny, 2: nx, 3: nx}
    edges = {0: (f[:, :, 0], f[:, :, -1]), 1: (f[:, :, -1], f[:, :, 0]), 2: (f[:, 0], f[:, -1]), 3: (f[:, -1], f[:, 0])}
    ghosts = []
    for k in range(4):
        side, (near, far) = p.sides[k], edges[k]
        along = (torch.arange(lens[k], dtype=torch.float64, device=f.device) + 0.5) * p.dx
        got = []
        for kind, state in ((side.kind_lo, side.state_lo), (side.kind_hi, side.state_hi)):
            if kind == "periodic":
                got.append(far)
            elif kind == "outflow":
                got.append(near)
            elif kind == "reflect":
                got.append(near[MIRROR_X if k < 2 else MIRROR_Y])
            else:
                q = [torch.tensor(float(v), dtype=torch.float64, device=f.device) for v in state]
                got.append(_equilibrium(s, *q)[:, None].expand(9, lens[k]))
        ghosts.append(torch.where(_part(side, along, t)[None], got[0], got[1]))
    left, right, bottom, top = ghosts
    return (torch.cat([f[:, :, 1:], right[:, :, None]], 2), torch.cat([left[:, :, None], f[:, :, :-1]], 2),
            torch.cat([f[:, 1:], top[:, None]], 1), torch.cat([bottom[:, None], f[:, :-1]], 1))


def _advance(s, f, E, Wt, N, S):
    fe = _equilibrium(s, *_moments(s, f))
    out = []
    for i in range(9):
        c, e, w, n, so = s.adv[i]
        out.append(f[i] + c * f[i] + e * E[i] + w * Wt[i] + n * N[i] + so * S[i] + s.omega * (fe[i] - f[i]))
    return torch.stack(out)


def _step(p, s, f, level):
    return _advance(s, f, *_neighbours(p, s, f, level))


def _totals(s, f):
    rho, ux, uy, T = _moments(s, f)
    return np.array([float(q.sum()) for q in (rho, rho * ux, rho * uy, rho * (s.b * T + ux * ux + uy * uy))])


def _names(q):
    return dict(zip(("rho", "ux", "uy", "T"), q))


@torch.no_grad()
def _exact_run(case, seed):
    p, given = _inputs(case, seed)
    s = _Scheme(p)
    if case["kind"] == "readout":
        f = given.double()
        return {**_names(_moments(s, f)), "totals": _totals(s, f), "f": f}
    f = _equilibrium(s, *[a.double() for a in given])
    totals, level = [], 0
    for _ in range(case.get("frames", 1)):
        for _ in range(case["steps"]):
            f = _step(p, s, f, level)
            level += 1
        totals.append(_totals(s, f))
    out = _names(_moments(s, f))
    return {"totals": np.stack(totals), **out} if case["kind"] == "watch" else out


@torch.no_grad()
def _exact_batch(case, seed):
    """All tubes side by side: periodic in y, outflow at each tube's ends."""
    probs, given = _inputs(case, seed)
    s = _Scheme(probs)
    f = _equilibrium(s, *[torch.cat([g[q].double() for g in given], 1) for q in range(4)])
    ends = np.cumsum([q.nx for q in probs])
    col = torch.arange(int(ends[-1]), device=DEV)
    last = torch.as_tensor(ends - 1, device=DEV)
    first = torch.as_tensor(np.concatenate([[0], ends[:-1]]), device=DEV)
    east, west = col + 1, col - 1
    east[last], west[first] = last, first
    for _ in range(case["steps"]):
        f = _advance(s, f, f[:, :, east], f[:, :, west], torch.roll(f, -1, 1), torch.roll(f, 1, 1))
    sizes = [q.nx for q in probs]
    return _names([torch.cat([b.reshape(-1) for b in a.split(sizes, 1)]) for a in _moments(s, f)])


def _exact_grad(case, seed):
    p, (fields, target) = _inputs(case, seed)
    tau = torch.tensor(float(torch.tensor(p.tau, dtype=_dtype(case))), dtype=torch.float64, requires_grad=True)
    fields = [a.double().requires_grad_(True) for a in fields]
    f = _equilibrium(_Scheme(p), *fields)
    for level in range(case["steps"]):
        f = checkpoint(lambda g, t, n=level: _step(p, _Scheme(p, t.to(g.device)), g, n), f, tau, use_reentrant=False)
    out = _moments(_Scheme(p), f)
    loss = 0.5 * torch.sum((out[0] - target.double()) ** 2)
    grads = torch.autograd.grad(loss, [*fields, tau])
    return {"out": [a.detach() for a in out], "grads": list(grads)}


def _exact_vn(case, seed):
    """max |eig G| with G = diag(symbol of the update) + omega df^eq/df, the
    Jacobian of the equilibrium by complex steps."""
    _, given = _inputs(case, seed)
    radius = np.empty((len(given), len(DIRS), NK))
    k = np.pi * np.arange(NK) / (NK - 1)
    for n, (p, q) in enumerate(given):
        s = _Scheme(p)
        vx, vy = np.array([float(v) for v in s.vx]), np.array([float(v) for v in s.vy])
        rho, ux, uy, T = q
        dF, h = np.empty((9, 4)), 1e-30
        for m in range(4):
            z = [torch.tensor(complex(v), dtype=torch.complex128) for v in q]
            z[m] = z[m] + 1j * h
            dF[:, m] = _equilibrium(s, *z).imag.numpy() / h
        eta = np.array([s.eta ** 2] + [0.0] * 8)
        dq = np.stack([np.ones(9), (vx - ux) / rho, (vy - uy) / rho,
                       ((vx - ux) ** 2 + (vy - uy) ** 2 + eta - p.b * T) / (p.b * rho)])
        G = np.broadcast_to(s.omega * (dF @ dq), (len(DIRS), NK, 9, 9)).astype(complex)
        for i in range(9):
            c, e, w, no, so = s.adv[i]
            for d, (dx, dy) in enumerate(DIRS):
                G[d, :, i, i] += (1.0 - s.omega + c + e * np.exp(1j * dx * k) + w * np.exp(-1j * dx * k)
                                  + no * np.exp(1j * dy * k) + so * np.exp(-1j * dy * k))
        radius[n] = np.abs(np.linalg.eigvals(G)).max(-1)
    return {"radius": torch.tensor(radius), "growth": torch.tensor(radius.max((1, 2)))}


def exact(case, seed):
    kind = case["kind"]
    if kind == "vn":
        return _exact_vn(case, seed)
    if kind == "batch":
        return _exact_batch(case, seed)
    if kind == "grad":
        return _exact_grad(case, seed)
    return _exact_run(case, seed)
