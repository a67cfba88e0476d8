"""Workloads that the solver is timed on, each through its public Python calls.

One pass of a case is what a program does with a problem in hand: set the initial fields, run the steps
(or the forward and backward pass of a gradient), read the result back on the device.  The kinds:

  tube      one 1-D shock tube (D1Q2 or D1Q3) with transmissive ends, to a final time
  quadrant  2-D four-quadrant Riemann problem, transmissive sides
  pulses    2-D uniform flow with Gaussian pulses, periodic sides
  oblique   2-D oblique-shock reflection: inflow, held top state, free-slip wall, outflow
  channel   Mach 3 channel with a forward-facing step (internal walls)
  burgers   scalar 2-D Burgers problem with boundary profiles
  tubes     many 1-D shock tubes of uneven length in one batched run
  gradient  gradient of a terminal density mismatch with respect to the initial fields (autograd)
  adaptive  quadrant problem with the lattice speed chosen every step, to an exact final time

`exact` computes the same results in FP64 with plain torch operations, without this package's library.
"""
import math
import random

import numpy as np
import torch
from torch.utils.checkpoint import checkpoint

from paper_1504_07034_gb300 import autograd
from paper_1504_07034_gb300.solver import BatchSolver, Solver

GAMMA = 1.4
INFLOW = (1.0, 2.9, 0.0, 1.0 / 1.4)                       # oblique shock: Mach 2.9
POST_SHOCK = (1.69997, 2.61934, -0.50632, 1.52819)        # behind its 29-degree shock
CHANNEL_INFLOW = (1.4, 3.0, 0.0, 1.0)                     # Mach 3
BURGERS = (1.0, -1.0, (1.0, -2.0))                        # left, right, bottom profile


def listed():
    return [
        # Sod's tube as the paper scales it: 1000 cells, FP64, a run of dependent small steps
        {"name": "tube_1000_f64", "kind": "tube", "nx": 1000, "steps": 461, "lattice": "d1q2",
         "precision": "f64", "omega": 1.0},
        # the paper's scalar problem on its own 64 x 64 grid to its steady state: the smallest 2-D run
        {"name": "burgers_64_f32", "kind": "burgers", "nx": 64, "ny": 64, "steps": 422, "precision": "f32"},
        # the benchmark configuration: 1024 x 1024 quadrant problem, 1000 FP32 steps
        {"name": "quadrant_1024_f32", "kind": "quadrant", "nx": 1024, "ny": 1024, "steps": 1000,
         "precision": "f32", "omega": 1.0},
        # the same grid on the FP64 path, which accuracy studies compare with
        {"name": "quadrant_1024_f64", "kind": "quadrant", "nx": 1024, "ny": 1024, "steps": 100,
         "precision": "f64", "omega": 1.0},
        # moments-only storage on a ragged grid (neither side a multiple of a tile)
        {"name": "quadrant_1531x973_f32u", "kind": "quadrant", "nx": 1531, "ny": 973, "steps": 400,
         "precision": "f32u", "omega": 1.0},
        # the large steady-flow run with mixed sides, its totals checked between chunks of steps
        {"name": "oblique_4096x1024_f32", "kind": "oblique", "nx": 4096, "ny": 1024, "steps": 600,
         "precision": "f32", "omega": 1.0},
        # the same flow with half-precision non-equilibrium parts, over-relaxed (where those parts matter)
        {"name": "oblique_2048x512_f16neq", "kind": "oblique", "nx": 2048, "ny": 512, "steps": 300,
         "precision": "f16neq", "omega": 1.5},
        # over-relaxed smooth flow (low numerical diffusion) on an odd grid: the full collision
        {"name": "pulses_1001x777_f32_w15", "kind": "pulses", "nx": 1001, "ny": 777, "steps": 300,
         "precision": "f32", "omega": 1.5},
        # internal walls: the forward-facing step, refined four times from the paper's 240 x 80
        {"name": "channel_960x320_f32", "kind": "channel", "nx": 960, "ny": 320, "steps": 400,
         "precision": "f32", "omega": 1.0},
        # parameter study: thousands of tubes of uneven length to one final time
        {"name": "tubes_4096_f32", "kind": "tubes", "count": 4096, "n_min": 200, "n_max": 20000,
         "t_final": 0.1, "lattice": "d1q2", "precision": "f32", "omega": 1.0},
        # inverse problem: forward and backward pass with sqrt(T) checkpoints
        {"name": "gradient_1024_f32", "kind": "gradient", "nx": 1024, "ny": 1024, "steps": 400,
         "precision": "f32", "omega": 1.0},
        # lattice speed taken from the flow at every step, exact final time
        {"name": "adaptive_768_f32", "kind": "adaptive", "nx": 768, "ny": 768, "steps": 384,
         "precision": "f32", "omega": 1.0},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """Two sides with the cell count between lo^2 and hi^2, up to 4 : 1, odd ones among them."""
    n, r = _log_int(rng, lo, hi), math.exp(rng.uniform(-math.log(2.0), math.log(2.0)))
    sides = [max(8, int(round(n * r))), max(8, int(round(n / r)))]
    return [s if rng.random() < 0.5 else max(8, s // 32 * 32) for s in sides]


def draw(rng):
    kind = rng.choice(["tube", "quadrant", "pulses", "oblique", "channel", "burgers", "tubes", "gradient", "adaptive"])
    if kind == "tube":
        lattice = rng.choice(["d1q2", "d1q3"])
        return {"kind": kind, "nx": _log_int(rng, 200, 20000), "steps": _log_int(rng, 100, 2000), "lattice": lattice,
                "precision": rng.choice(["f32", "f64"]), "omega": 1.0 if lattice == "d1q3" else rng.choice([1.0, 1.3])}
    if kind == "tubes":
        return {"kind": kind, "count": _log_int(rng, 64, 2048), "n_min": 200, "n_max": _log_int(rng, 1000, 15000),
                "t_final": 0.1, "lattice": rng.choice(["d1q2", "d1q3"]), "precision": "f32", "omega": 1.0}
    if kind == "channel":
        ny = 10 * _log_int(rng, 4, 64)
        return {"kind": kind, "nx": 3 * ny, "ny": ny, "steps": rng.randint(60, 500), "precision": "f32", "omega": 1.0}
    if kind == "burgers":
        nx, ny = _grid(rng, 48, 3000)
        return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(60, 500), "precision": "f32"}
    if kind == "gradient":
        nx, ny = _grid(rng, 48, 1200)
        return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(30, 300),
                "precision": rng.choice(["f32", "f32", "f32", "f64"]), "omega": rng.choice([1.0, 1.0, 1.5])}
    if kind == "adaptive":
        nx, ny = _grid(rng, 64, 1200)
        return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(80, 400),
                "precision": rng.choice(["f32", "f32", "f64"]), "omega": 1.0}
    precision = rng.choice(["f32", "f32", "f32", "f32u", "f64", "f16neq"])
    nx, ny = _grid(rng, 64, 900 if precision == "f64" else 2400)
    omega = 1.0 if precision == "f32u" or kind == "quadrant" else rng.choice([1.0, 1.5])
    return {"kind": kind, "nx": nx, "ny": ny, "steps": rng.randint(40, 100 if precision == "f64" else 500),
            "precision": precision, "omega": omega}


# ---------------------------------------------------------------- inputs

def _sound(rho, p):
    return math.sqrt(GAMMA * p / rho)


def _speed2d(rho, u, v, p):
    return abs(u) + abs(v) + math.sqrt(2.0) * _sound(rho, p)


def _star(left, right):
    """Exact solution of the Riemann problems left | right, arrays of (rho, u, p) each: the velocity
    between the waves and the densities and the pressure there; whether vacuum would form (the values
    mean nothing then)."""
    g, sides = (GAMMA - 1.0) / (GAMMA + 1.0), (left, right)
    a = [np.sqrt(GAMMA * w[2] / w[0]) for w in sides]

    def jump(p, w, s):                            # velocity change across the wave of one side
        shock = (p - w[2]) * np.sqrt(2.0 / ((GAMMA + 1.0) * w[0]) / (p + g * w[2]))
        fan = 2.0 * s / (GAMMA - 1.0) * ((p / w[2]) ** ((GAMMA - 1.0) / (2.0 * GAMMA)) - 1.0)
        return np.where(p > w[2], shock, fan)

    lo, hi = np.full_like(a[0], -40.0), np.full_like(a[0], 8.0)        # logarithm of the pressure
    for _ in range(70):
        mid = 0.5 * (lo + hi)
        up = jump(np.exp(mid), left, a[0]) + jump(np.exp(mid), right, a[1]) + right[1] - left[1] < 0.0
        lo, hi = np.where(up, mid, lo), np.where(up, hi, mid)
    p = np.exp(0.5 * (lo + hi))
    u = 0.5 * (left[1] + right[1]) + 0.5 * (jump(p, right, a[1]) - jump(p, left, a[0]))
    rho = [np.where(p > w[2], w[0] * (p / w[2] + g) / (g * p / w[2] + 1.0), w[0] * (p / w[2]) ** (1.0 / GAMMA))
           for w in sides]
    return u, rho[0], rho[1], p, 2.0 / (GAMMA - 1.0) * (a[0] + a[1]) <= right[1] - left[1]


def _speed1d(left, right):
    """Largest |u| + a over the constant states of the solutions left | right, and whether vacuum forms."""
    u, rl, rr, p, vacuum = _star(left, right)
    c = [np.abs(w[1]) + np.sqrt(GAMMA * w[2] / w[0]) for w in (left, right)]
    c += [np.abs(u) + np.sqrt(GAMMA * p / r) for r in (rl, rr)]
    return np.max(c, axis=0), vacuum


def _quadrants(rng):
    """States (rho, u, v, p) of the four quadrants, counter-clockwise from the top right, and the lattice
    speed: above the D2Q4 bound of every constant state of the four interface problems."""
    while True:
        q = [(rng.uniform(0.1, 1.5), rng.uniform(-1.2, 1.2), rng.uniform(-1.2, 1.2), rng.uniform(0.03, 1.5))
             for _ in range(4)]
        lam, bad = max(_speed2d(*s) for s in q), False
        for a, b, normal in ((1, 0, 1), (2, 3, 1), (3, 0, 2), (2, 1, 2)):
            left, right = (np.array([[q[s][0]], [q[s][normal]], [q[s][3]]]) for s in (a, b))
            u, rl, rr, p, vacuum = (float(v[0]) for v in _star(left, right))
            bad |= bool(vacuum)
            lam = max(lam, *(_speed2d(r, u, q[s][3 - normal], p) for r, s in ((rl, a), (rr, b))))
        if not bad:
            return q, 1.1 * lam


def _bumps(rng, nx, ny, amp, count=8, width=0.05):
    """(ny, nx) sum of Gaussian bumps on the periodic unit-height box, cells of side 1 / ny."""
    x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / ny
    y = (torch.arange(ny, dtype=torch.float64, device="cuda") + 0.5) / ny
    length, f = nx / ny, torch.zeros(ny, nx, dtype=torch.float64, device="cuda")
    for _ in range(count):
        dx, dy = (x - length * rng.random()).abs(), (y - rng.random()).abs()
        dx, dy = torch.minimum(dx, length - dx), torch.minimum(dy, 1.0 - dy)
        f += amp * torch.exp(-dy ** 2 / (2 * width ** 2))[:, None] * torch.exp(-dx ** 2 / (2 * width ** 2))[None, :]
    return f


def _uniform(state, nx, ny):
    return torch.tensor(state, dtype=torch.float64, device="cuda")[:, None, None].expand(-1, ny, nx).clone()


def _problem(case, seed):
    """Fields, sides, lattice speed and the rest of a 1-D or 2-D problem on one grid."""
    rng = random.Random(seed)
    kind, nx, ny = case["kind"], case["nx"], case.get("ny", 1)
    p = {"dx": 1.0 / ny, "solid": None, "omega": case.get("omega", 1.0)}
    if kind == "tube":
        left = (rng.uniform(0.9, 1.1), 0.0, rng.uniform(0.9, 1.1))
        right = (0.125 * rng.uniform(0.9, 1.1), 0.0, 0.1 * rng.uniform(0.9, 1.1))
        x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx
        ends = torch.tensor([left, right], dtype=torch.float64, device="cuda")
        W = torch.where((x < 0.5)[None, :], ends[0][:, None], ends[1][:, None])
        lam = 2.4 * (math.sqrt(1.5) if case["lattice"] == "d1q3" else 1.0)   # above |u| + a of the solution
        return dict(p, W=W, dx=1.0 / nx, lam=lam, bc=[("transmissive", None)] * 2)
    if kind in ("quadrant", "adaptive"):
        q, lam = _quadrants(rng)
        right = (torch.arange(nx, device="cuda") >= nx // 2)[None, :]
        top = (torch.arange(ny, device="cuda") >= ny // 2)[:, None]
        t = torch.tensor(q, dtype=torch.float64, device="cuda")
        which = torch.where(top, torch.where(right, 0, 1), torch.where(right, 3, 2))
        W = t[which].permute(2, 0, 1).contiguous()
        return dict(p, W=W, lam=lam, bc=[("transmissive", None)] * 4)
    if kind in ("pulses", "gradient"):
        W = _uniform((1.0, 0.5, 0.3, 1.0), nx, ny)
        bump = _bumps(rng, nx, ny, 0.1)
        W[0] += bump
        W[3] += bump
        if kind == "gradient":
            p["target"] = 1.0 + _bumps(rng, nx, ny, 0.1)
        return dict(p, W=W, lam=3.0, bc=[("periodic", None)] * 4)
    if kind == "oblique":
        W = _uniform(INFLOW, nx, ny)
        bump = _bumps(rng, nx, ny, 0.05)
        W[0] += bump
        W[3] += bump
        bc = [("dirichlet", INFLOW), ("transmissive", None), ("wall", None), ("dirichlet", POST_SHOCK)]
        return dict(p, W=W, lam=1.15 * max(_speed2d(*INFLOW), _speed2d(*POST_SHOCK)), bc=bc)
    if kind == "channel":
        W = _uniform(CHANNEL_INFLOW, nx, ny)
        bump = _bumps(rng, nx, ny, 0.05)
        W[0] += bump
        W[3] += bump
        x = (torch.arange(nx, device="cuda") + 0.5) / ny
        y = (torch.arange(ny, device="cuda") + 0.5) / ny
        p["solid"] = ((x >= 0.6)[None, :] & (y < 0.2)[:, None]).to(torch.uint8)
        bc = [("dirichlet", CHANNEL_INFLOW), ("transmissive", None), ("wall", None), ("wall", None)]
        return dict(p, W=W, lam=6.65, bc=bc)          # 1.5 x the bound behind a standing Mach 3 shock
    if kind == "burgers":
        left, right, (b0, b1) = BURGERS
        x = (torch.arange(nx, dtype=torch.float64, device="cuda") + 0.5) / nx
        W = (b0 + b1 * x)[None, None, :] + 0.2 * _bumps(rng, nx, ny, 1.0)[None].clamp(max=1.0)
        bc = [("dirichlet", (left, 0.0, 0.0, 0.0)), ("dirichlet", (right, 0.0, 0.0, 0.0)),
              ("dirichlet", (b0, b1, 0.0, 0.0)), ("transmissive", None)]
        return dict(p, W=W, dx=1.0 / nx, lam=2.5, bc=bc)
    raise ValueError(kind)


def _tubes(case, seed):
    """Lengths, end states, lattice speeds and steps of a batch of tubes (host arrays).  The lengths are
    those of the study (the same for every seed), the states and with them the steps the seed's."""
    B = case["count"]
    n = np.random.default_rng(B).uniform(math.log(case["n_min"]), math.log(case["n_max"]), B)
    n = np.rint(np.exp(n)).astype(np.int64)
    rng = np.random.default_rng(seed)
    d = rng.uniform(size=(6, B))
    left = np.stack([0.05 + 1.95 * d[0], -1.0 + 2.0 * d[1], 0.05 + 1.95 * d[2]])
    right = np.stack([0.05 + 1.95 * d[3], -1.0 + 2.0 * d[4], 0.05 + 1.95 * d[5]])
    right[1] = np.where(_speed1d(left, right)[1], left[1], right[1])          # no vacuum
    lam = 1.05 * _speed1d(left, right)[0]
    lam *= math.sqrt(1.5) if case["lattice"] == "d1q3" else 1.0
    steps = np.ceil(case["t_final"] * lam * n).astype(np.int64)
    lam = steps / (case["t_final"] * n)                             # whole steps to the final time
    return n, left, right, lam, steps


def _tubes_fields(n, left, right):
    """Concatenated primitive fields (3, sum n) on the GPU."""
    lengths = torch.from_numpy(n).cuda()
    tube = torch.repeat_interleave(torch.arange(len(n), device="cuda"), lengths)
    start = torch.cumsum(lengths, 0) - lengths
    first = torch.arange(len(tube), device="cuda") - start[tube] < (lengths[tube] + 1) // 2
    return torch.where(first, torch.from_numpy(left).cuda()[:, tube], torch.from_numpy(right).cuda()[:, tube])


def _dtype(case):
    return torch.float64 if case["precision"] == "f64" else torch.float32


def prepare(case, seed):
    if case["kind"] == "tubes":
        n, left, right, lam, steps = _tubes(case, seed)
        s = BatchSolver(n, lam, omega=case["omega"], precision=case["precision"], lattice=case["lattice"])
        return {"case": case, "solver": s, "W": _tubes_fields(n, left, right), "steps": steps}
    p = _problem(case, seed)
    kind = case["kind"]
    lattice = case["lattice"] if kind == "tube" else ("d2q4s" if kind == "burgers" else "d2q4")
    s = Solver(lattice, case["nx"], case.get("ny", 1), lam=p["lam"], dx=p["dx"], bc=p["bc"], gamma=GAMMA,
               omega=p["omega"], precision=case["precision"])
    if p["solid"] is not None:
        s.set_obstacles(p["solid"])
    state = {"case": case, "solver": s, "W": p["W"]}
    if kind == "gradient":
        s.set_state(p["W"])
        state["U0"] = s.moments(dtype=_dtype(case)).requires_grad_()
        state["target"] = p["target"].to(_dtype(case))
    if kind == "adaptive":
        state["t_final"] = case["steps"] * p["dx"] / p["lam"]
    return state


def run(state):
    case, s = state["case"], state["solver"]
    kind, out = case["kind"], _dtype(case)
    if kind == "gradient":
        U = autograd.run(state["U0"], s, case["steps"])
        loss = 0.5 * ((U[0] - state["target"]) ** 2).sum()
        (grad,) = torch.autograd.grad(loss, state["U0"])
        return {"U": U.detach(), "loss": loss.detach(), "grad": grad}
    s.set_state(state["W"])
    if kind == "tubes":
        s.run(state["steps"])
        return s.moments(dtype=out)
    if kind == "adaptive":
        st = s.run_to_time(state["t_final"], safety=1.05)
        return {"U": s.moments(dtype=out), "t": st["t"], "lambda": st["lambda"], "steps": st["steps"]}
    if kind == "oblique":                       # totals and bounds in FP64 after each third of the run
        checks, done = [], 0
        for part in (1, 2, 3):
            n = case["steps"] * part // 3 - done
            s.step(n)
            done += n
            d = s.diagnostics()
            checks.append(d["totals"] + [d["min_rho"], d["min_p"], d["max_lambda_local"]])
        return {"U": s.moments(dtype=out), "checks": np.array(checks, dtype=np.float32),
                "bad": np.array([d["n_nonphysical"], d["n_subchar"]])}
    s.step(case["steps"])
    return s.moments(dtype=out)


# ---------------------------------------------------------------- work

# Floating-point operations of one lattice update at omega = 1, as the method states them: the moment
# sums, velocities, pressure, fluxes and equilibria of each field (FP64 and FP32 alike).
UPDATE_FLOPS = {"d2q4": 74, "d2q4s": 15, "d1q2": 24, "d1q3": 27}


def work(case):
    """Inputs read once, outputs written once; the steps' state can stay on the chip's caches only
    where it fits, so no traffic between steps is counted."""
    kind = case["kind"]
    ob = 8 if case["precision"] == "f64" else 4
    if kind == "tubes":
        n, _, _, _, steps = _tubes(case, 0)
        return {"bytes": float(n.sum()) * 3 * (8 + ob), "flops": float((n * steps).sum()) * UPDATE_FLOPS[case["lattice"]]}
    cells = case["nx"] * case.get("ny", 1)
    if kind == "tube":
        lattice, fields = case["lattice"], 3
    elif kind == "burgers":
        lattice, fields = "d2q4s", 1
    else:
        lattice, fields = "d2q4", 4
    flops = UPDATE_FLOPS[lattice] * float(cells) * case["steps"]
    if case.get("omega", 1.0) != 1.0:          # relaxation of each population: two products and a sum
        flops *= 1.0 + 3.0 * fields * {"d1q2": 2, "d1q3": 3}.get(lattice, 4) / UPDATE_FLOPS[lattice]
    if kind == "gradient":                     # forward, recomputed forward, adjoint (about twice a step)
        return {"bytes": float(cells) * (4 * ob * 3 + ob), "flops": 4.0 * flops}
    return {"bytes": float(cells) * fields * (8 + ob), "flops": flops}


# ---------------------------------------------------------------- the same results in FP64, plain torch

SX, SY = (-1, 1, 1, -1), (-1, -1, 1, 1)


def _cons2d(W):
    rho, u, v, p = W
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)])


def _feq2d(U, c):
    rho, mx, my, en = U
    u, v = mx / rho, my / rho
    p = (GAMMA - 1.0) * (en - 0.5 * (mx * u + my * v))
    a, F, G = 0.25 * U, c * torch.stack([mx, mx * u + p, mx * v, u * (en + p)]), \
        c * torch.stack([my, my * u, my * v + p, v * (en + p)])
    return torch.stack([a - F - G, a + F - G, a + F + G, a - F + G])


def _feq2ds(u, c):
    a, F, G = 0.25 * u, c * (0.5 * u * u), c * u
    return torch.stack([a - F - G, a + F - G, a + F + G, a - F + G])


def _pad2d(f, bc, ghost, axis):
    """f (..., ny, nx) with one more row (axis -2) or column (axis -1) at each end, by the sides' kinds;
    ghost[s] broadcasts against the added slice."""
    lo, hi = (2, 3) if axis == -2 else (0, 1)
    n = f.shape[axis]
    ends = []
    for s, (at, wrapped) in ((lo, (0, n - 1)), (hi, (n - 1, 0))):
        e = f.narrow(axis, wrapped if bc[s][0] == "periodic" else at, 1)
        ends.append(ghost[s].expand_as(e) if bc[s][0] == "dirichlet" else e)
    return torch.cat([ends[0], f, ends[1]], axis)


def _ghosts2d(bc, c):
    return {s: _feq2d(_cons2d(torch.tensor(b[1], dtype=torch.float64, device="cuda")), c)[:, :, None, None]
            for s, b in enumerate(bc) if b[0] == "dirichlet"}


def _ghosts2ds(bc, c, nx, ny, dx):
    g = {}
    for s, b in enumerate(bc):
        if b[0] == "dirichlet":
            m = torch.arange(-1, ny + 1) if s < 2 else torch.arange(nx)
            e = _feq2ds(b[1][0] + b[1][1] * (m.double().cuda() + 0.5) * dx, c)[:, None]
            g[s] = e[..., :, None] if s < 2 else e[..., None, :]
    return g


def _stream2d(f, bc, ghost, walls=None):
    """Pulled populations of f (4, K, ny, nx)."""
    ny, nx = f.shape[-2:]
    p = _pad2d(_pad2d(f, bc, ghost, -2), bc, ghost, -1)
    g = [p[q][..., 1 - SY[q]:1 - SY[q] + ny, 1 - SX[q]:1 - SX[q] + nx] for q in range(4)]
    if walls is not None:
        solid, rules = walls
        out = []
        for q in range(4):
            v = g[q]
            for m, su, sv, where in rules[q]:
                sign = torch.tensor([1.0, su, sv, 1.0], dtype=torch.float64, device="cuda")[:, None, None]
                v = torch.where(where, sign * g[m], v)
            out.append(v)
        g = out
    g = torch.stack(g)
    flip = torch.tensor([1.0, 1.0, -1.0, 1.0], dtype=torch.float64, device="cuda")[: f.shape[1], None]
    if bc[3][0] == "wall":
        g[0, :, -1], g[1, :, -1] = flip * g[3, :, -1], flip * g[2, :, -1]
    if bc[2][0] == "wall":
        g[3, :, 0], g[2, :, 0] = flip * g[0, :, 0], flip * g[1, :, 0]
    return g


def _wall_rules(solid, bc):
    """Per population: (mirror population, sign of rho u, sign of rho v, cells) of the internal walls."""
    zero = {s: torch.zeros((), dtype=solid.dtype, device="cuda") for s in range(4)}
    as_fluid = [(("dirichlet", None) if b[0] in ("dirichlet", "wall") else b) for b in bc]
    p = _pad2d(_pad2d(solid[None], as_fluid, zero, -2), as_fluid, zero, -1)[0].bool()
    ny, nx = solid.shape
    at = lambda dx, dy: p[1 + dy:1 + dy + ny, 1 + dx:1 + dx + nx]  # noqa: E731
    rules = []
    for q in range(4):
        src, xn, yn = at(-SX[q], -SY[q]), at(-SX[q], 0), at(0, -SY[q])
        unknown = src & ~solid.bool()
        pop = {(SX[m], SY[m]): m for m in range(4)}
        rules.append([(pop[-SX[q], SY[q]], -1.0, 1.0, unknown & xn & ~yn),
                      (pop[SX[q], -SY[q]], 1.0, -1.0, unknown & yn & ~xn),
                      (pop[-SX[q], -SY[q]], -1.0, -1.0, unknown & (xn == yn))])
    return solid.bool(), rules


def _step2d(f, bc, ghost, c, om, walls=None):
    g = _stream2d(f, bc, ghost, walls)
    new = om * _feq2d(g.sum(0), c) + (1.0 - om) * g if om != 1.0 else _feq2d(g.sum(0), c)
    return torch.where(walls[0], f, new) if walls is not None else new


def _speeds(U):
    rho, mx, my, en = U
    u, v = mx / rho, my / rho
    p = (GAMMA - 1.0) * (en - 0.5 * (mx * u + my * v))
    return torch.maximum((u + v).abs(), (u - v).abs()) + math.sqrt(2.0) * torch.sqrt(GAMMA * p / rho), p


def _exact_check(f, dx):
    U = f.sum(0)
    s, p = _speeds(U)
    tot = U.sum((1, 2)) * dx * dx
    return torch.cat([tot, torch.stack([U[0].min(), p.min(), s.max()])]).cpu().numpy()


def _exact_adaptive(case, p):
    dx, lam, t_final = p["dx"], p["lam"], case["steps"] * p["dx"] / p["lam"]
    f = _feq2d(_cons2d(p["W"]), 1.0 / (4.0 * lam))
    t, steps, last, done = 0.0, 0, False, False
    while not done:
        # the step streams with lam and collides with the speed chosen from the state before it
        bound = float(_speeds(f.sum(0))[0].max())
        t_next = t_final if last else t + dx / lam
        new, next_last = 1.05 * bound, False
        if not last and t_next + dx / new >= t_final:
            new, next_last = dx / (t_final - t_next), True
        f = _step2d(f, p["bc"], {}, 1.0 / (4.0 * new), 1.0)
        t, lam, steps, done, last = t_next, new, steps + 1, last, next_last
    return {"U": f.sum(0), "t": t, "lambda": lam, "steps": None}


def _exact_gradient(case, p):
    c, om, bc, n = 1.0 / (4.0 * p["lam"]), p["omega"], p["bc"], case["steps"]
    U0 = _cons2d(p["W"])
    if case["precision"] != "f64":
        U0 = U0.float().double()                  # the values that the solver is given
    U0.requires_grad_()

    def some(f, m):
        for _ in range(m):
            f = _step2d(f, bc, {}, c, om)
        return f

    f = _feq2d(U0, c)
    seg = max(1, min(int(math.sqrt(n)), int(2e8 / (case["nx"] * case["ny"] * 16))))
    for m0 in range(0, n, seg):
        f = checkpoint(some, f, min(seg, n - m0), use_reentrant=False)
    U = f.sum(0)
    target = p["target"].to(_dtype(case)).double()
    loss = 0.5 * ((U[0] - target) ** 2).sum()
    (grad,) = torch.autograd.grad(loss, U0)
    return {"U": U.detach(), "loss": loss.detach(), "grad": grad}


def _cons1d(W):
    rho, u, p = W
    return torch.stack([rho, rho * u, p / (GAMMA - 1.0) + 0.5 * rho * u * u])


def _feq1d(U, c, lattice):
    rho, m, en = U
    u = m / rho
    p = (GAMMA - 1.0) * (en - 0.5 * m * u)
    G = c * torch.stack([m, m * u + p, u * (en + p)])
    if lattice == "d1q3":
        return torch.stack([U / 3.0 - G, U / 3.0, U / 3.0 + G])
    return torch.stack([0.5 * U - G, 0.5 * U + G])


def _step1d(f, first, last, c, om, lattice):
    """One step of tubes side by side; first, last: the end cells (an end pulls its own value)."""
    up, down = f[0].roll(-1, 1), f[-1].roll(1, 1)
    up[:, last], down[:, first] = f[0][:, last], f[-1][:, first]
    g = torch.stack([up, f[1], down] if lattice == "d1q3" else [up, down])
    e = _feq1d(g.sum(0), c, lattice)
    return e if om == 1.0 else (1.0 - om) * g + om * e


def _exact_tubes(case, seed):
    n, left, right, lam, steps = _tubes(case, seed)
    order = np.argsort(-steps, kind="stable")                 # the tubes still running are a prefix
    ns, ss = n[order], steps[order]
    f_lam = torch.repeat_interleave(torch.from_numpy(lam[order]).cuda(), torch.from_numpy(ns).cuda())
    end = np.cumsum(ns)
    first, last = torch.from_numpy(end - ns).cuda(), torch.from_numpy(end - 1).cuda()
    c = 1.0 / (2.0 * f_lam)
    f = _feq1d(_cons1d(_tubes_fields(ns, left[:, order], right[:, order])), c, case["lattice"])
    for k in range(int(ss[0])):
        t = int(np.searchsorted(-ss, -k))                     # tubes with more than k steps
        m = int(end[t - 1])
        f[:, :, :m] = _step1d(f[:, :, :m], first[:t], last[:t], c[:m], case["omega"], case["lattice"])
    U, out = f.sum(0), torch.empty(3, int(end[-1]), dtype=torch.float64, device="cuda")
    starts = np.cumsum(n) - n
    for b, (e, m) in enumerate(zip(end, ns)):
        out[:, starts[order[b]]:starts[order[b]] + m] = U[:, e - m:e]
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "tubes":
        return _exact_tubes(case, seed)
    p = _problem(case, seed)
    om, lam = p["omega"], p["lam"]
    if kind == "tube":
        c = 1.0 / (2.0 * lam)
        f = _feq1d(_cons1d(p["W"]), c, case["lattice"])
        for _ in range(case["steps"]):
            f = _step1d(f, [0], [case["nx"] - 1], c, om, case["lattice"])
        return f.sum(0)
    if kind == "adaptive":
        return _exact_adaptive(case, p)
    if kind == "gradient":
        return _exact_gradient(case, p)
    c = 1.0 / (4.0 * lam)
    if kind == "burgers":
        ghost = _ghosts2ds(p["bc"], c, case["nx"], case["ny"], p["dx"])
        f = _feq2ds(p["W"], c)
        for _ in range(case["steps"]):
            f = _feq2ds(_stream2d(f, p["bc"], ghost).sum(0), c)
        return f.sum(0)
    ghost = _ghosts2d(p["bc"], c)
    walls = _wall_rules(p["solid"], p["bc"]) if p["solid"] is not None else None
    f = _feq2d(_cons2d(p["W"]), c)
    checks = []
    for k in range(1, case["steps"] + 1):
        f = _step2d(f, p["bc"], ghost, c, om, walls)
        if kind == "oblique" and k in [case["steps"] * part // 3 for part in (1, 2, 3)]:
            checks.append(_exact_check(f, p["dx"]))
    if kind == "oblique":
        return {"U": f.sum(0), "checks": np.array(checks), "bad": None}
    return f.sum(0)
