"""Workloads of the library, each one pass through its public entry points.

A case says which entry point is called and on what: a right-hand side with its
stencil codes, a march (``run``) of a 1D or 2D system, a ragged batch of shock
tubes, a checkpointed gradient, or the call on host arrays.  ``prepare`` makes
the state a program has in hand (seeded initial data on the GPU, the context),
``run`` makes the call, ``exact`` computes the same result with plain torch
operations in 64 bits.
"""
import math

import numpy as np
import torch

from paper_1808_00037_gb300 import adjoint as A
from paper_1808_00037_gb300 import binding as B

GAMMA = 1.4
CT = 1e-5
PREC = {"f64": B.T7_F64, "f32": B.T7_F32, "mixed": B.T7_MIXED}
SYSTEM = {"advection": B.T7_SCALAR_ADVECTION, "burgers": B.T7_BURGERS, "euler1d": B.T7_EULER1D,
          "euler2d": B.T7_EULER2D}
FIELDS = {"advection": 1, "burgers": 1, "euler1d": 3, "euler2d": 4}
CFL = {"advection": 0.2, "burgers": 0.5, "euler1d": 0.5, "euler2d": 0.4}
# floating-point operations per cell and Runge-Kutta stage: staging, Roe frame,
# projection, smoothness measures, polynomials, back-projection, update
FLOPS = {"advection": 110, "burgers": 170, "euler1d": 800, "euler2d": 2200}
ADJOINT_FLOPS = 2000  # one adjoint stage per cell


def listed():
    return [
        # the smallest call: one right-hand side with its codes, as a dispersion analysis makes hundreds of
        {"name": "rhs-advection-f64-200", "kind": "rhs", "system": "advection", "prec": "f64", "n": 200},
        # one right-hand side with its codes of an ordinary ragged grid (parity checks, error studies)
        {"name": "rhs-euler1d-f32-100003", "kind": "rhs", "system": "euler1d", "prec": "f32", "n": 100003},
        # the advection accuracy run: sin(pi x), 200 cells, CFL 0.2, one period (about 1000 steps)
        {"name": "run-advection-f64-200", "kind": "run", "system": "advection", "prec": "f64", "n": 200,
         "steps": 2000, "t_end": 2.0},
        # the Shu-Osher case at its published 1600 cells, a stretch of the run to t = 1.8
        {"name": "run-euler1d-f64-1600", "kind": "run", "system": "euler1d", "prec": "f64", "n": 1600, "steps": 256},
        {"name": "run-euler1d-f32-1600", "kind": "run", "system": "euler1d", "prec": "f32", "n": 1600, "steps": 256},
        # the same profile repeated over a long domain: a bulk FP64 run and the largest FP32 one
        {"name": "run-euler1d-f64-1000003", "kind": "run", "system": "euler1d", "prec": "f64", "n": 1000003,
         "steps": 2},
        {"name": "run-euler1d-f32-16777600", "kind": "run", "system": "euler1d", "prec": "f32", "n": 16777600,
         "steps": 4},
        # 2D four-quadrant data: FP32 bulk with FP64 sums at the benchmark grid, and full FP64 on a ragged grid
        {"name": "run-euler2d-f32-2048x2048", "kind": "run", "system": "euler2d", "prec": "f32", "n": 2048,
         "ny": 2048, "steps": 4},
        {"name": "run-euler2d-f64-700x650", "kind": "run", "system": "euler2d", "prec": "f64", "n": 700, "ny": 650,
         "steps": 4},
        # ragged batches of Riemann tubes of 256 to 8192 cells: the 4096 tubes of the benchmark, 20 steps of each
        {"name": "batch-f32-4096", "kind": "batch", "prec": "f32", "tubes": 4096, "nmin": 256, "nmax": 8192,
         "steps": 20},
        # the gradient of the sine-mode problem through a checkpointed run (100 of its 2000 steps)
        {"name": "gradient-f64-4096", "kind": "gradient", "prec": "f64", "n": 4096, "steps": 100, "every": 50},
        # the call on a page-locked host array, one step a call (copy in, step, copy out)
        {"name": "host-euler1d-f32-4194301", "kind": "host", "system": "euler1d", "prec": "f32", "n": 4194301,
         "steps": 1},
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["rhs", "run", "run", "run", "run2d", "run2d", "batch", "gradient", "host"])
    prec = rng.choice(["f64", "f32"])
    if kind == "rhs":
        system = rng.choice(["advection", "burgers", "euler1d"])
        return {"kind": "rhs", "system": system, "prec": prec, "n": size(40, 2000000)}
    if kind == "run":
        system = rng.choice(["advection", "burgers", "euler1d", "euler1d"])
        prec = rng.choice(["f64", "f32", "mixed"])
        n = size(40, 1000003 if prec == "f64" else 16777600)
        # short domains are marched far, long ones a few steps
        return {"kind": "run", "system": system, "prec": prec, "n": n, "steps": max(1, min(256, 2000000 // n))}
    if kind == "run2d":
        prec = rng.choice(["f64", "f32", "mixed"])
        top = 700 if prec == "f64" else 2048
        nx, ny = size(40, top), size(40, top)
        return {"kind": "run", "system": "euler2d", "prec": prec, "n": nx, "ny": ny,
                "steps": max(1, min(64, 1000000 // (nx * ny)))}
    if kind == "batch":
        tubes = size(20, 4096 if prec == "f32" else 200)
        return {"kind": "batch", "prec": prec, "tubes": tubes, "nmin": 256, "nmax": 8192 if prec == "f32" else 2048,
                "steps": 20}
    if kind == "gradient":
        return {"kind": "gradient", "prec": prec, "n": size(200, 4500), "steps": rng.randint(10, 60),
                "every": rng.randint(5, 40)}
    return {"kind": "host", "system": "euler1d", "prec": prec, "n": size(1000, 4194301 if prec == "f32" else 500000),
            "steps": 1}


# ------------------------------------------------------------------ inputs --
def _periodic(case):
    """Periodic ends for smooth data, zero-gradient ends for shocks."""
    return case["kind"] == "gradient" or case["system"] in ("advection", "burgers")


def _dx(case):
    if case["kind"] == "gradient":
        return 1.0 / case["n"]
    if case["system"] in ("advection", "burgers"):
        return 2.0 / case["n"]
    if case["system"] == "euler1d":
        return 10.0 / min(case["n"], 1600)  # long domains repeat the Shu-Osher profile at its published width
    return 1.0 / case["n"]


def _euler1d(rho, u, p):
    return torch.stack([rho, rho * u, p / (GAMMA - 1.0) + 0.5 * rho * u * u])


def _state64(case, seed):
    """Initial data in 64 bits on the GPU."""
    g = np.random.default_rng(seed)
    n, dev = case["n"], "cuda"
    i = torch.arange(n, dtype=torch.float64, device=dev)
    if case["kind"] == "gradient":
        # rho = 1 + sum a_k sin(2 pi k x), a_k ~ N(0, (0.02/k)^2), u = p = 1 on periodic [0, 1)
        k = np.arange(1, 65)
        a = torch.tensor(g.normal(0.0, 1.0, 64) * (0.02 / k), device=dev)
        x = (i + 0.5) / n
        rho = 1.0 + torch.sin(2 * math.pi * torch.outer(x, torch.arange(1, 65, dtype=torch.float64, device=dev))) @ a
        return _euler1d(rho, torch.ones_like(rho), torch.ones_like(rho))
    system = case["system"]
    if system == "advection":
        return torch.sin(math.pi * ((i + 0.5) * (2.0 / n) - 1.0) + g.uniform(0, 2 * math.pi))[None].contiguous()
    if system == "burgers":
        return (0.5 + torch.sin(math.pi * (i + 0.5) * (2.0 / n) + g.uniform(0, 2 * math.pi)))[None].contiguous()
    if system == "euler1d":
        # Shu-Osher's shock and entropy wave on 1600 cells (or on all of a shorter domain), repeated
        period = min(n, 1600)
        amp, phase = g.uniform(0.18, 0.22), g.uniform(-0.5, 0.5)
        x = -5.0 + (torch.remainder(i, float(period)) + 0.5) * (10.0 / period)
        left = x < -4.0
        rho = torch.where(left, 3.857143, 1.0 + amp * torch.sin(5.0 * x + phase))
        u = torch.where(left, 2.629369, 0.0).double()
        p = torch.where(left, 10.33333, 1.0).double()
        return _euler1d(rho, u, p)
    # four quadrants, each its own constant state; no vacuum between neighbours
    ny = case["ny"]
    while True:
        q = np.stack([g.uniform(0.1, 1.5, 4), g.uniform(-1.2, 1.2, 4), g.uniform(-1.2, 1.2, 4),
                      g.uniform(0.03, 1.5, 4)])
        c = np.sqrt(GAMMA * q[3] / q[0])
        pairs = ((1, 0, 1), (2, 3, 1), (3, 0, 2), (2, 1, 2))
        if all(q[v][b] - q[v][a] < 5.0 * (c[a] + c[b]) for a, b, v in pairs):
            break
    right = ((i + 0.5) / n > 0.5)[None, :]
    top = ((torch.arange(ny, dtype=torch.float64, device=dev) + 0.5) / ny > 0.5)[:, None]
    quadrant = torch.where(right, torch.where(top, 0, 3), torch.where(top, 1, 2))
    rho, u, v, p = torch.tensor(q, device=dev)[:, quadrant]
    return torch.stack([rho, rho * u, rho * v, p / (GAMMA - 1.0) + 0.5 * rho * (u * u + v * v)]).contiguous()


def _tubes64(case, seed):
    """Concatenated Riemann tubes on [0, 1], jump at 0.5, and their lengths."""
    lengths = np.random.default_rng(7).integers(case["nmin"], case["nmax"] + 1, size=case["tubes"])
    g = np.random.default_rng(seed)
    s = torch.tensor(np.stack([g.uniform(0.1, 2.0, (2, case["tubes"])), g.uniform(-1.0, 1.0, (2, case["tubes"])),
                               g.uniform(0.1, 10.0, (2, case["tubes"]))]), device="cuda")
    length = torch.tensor(lengths, device="cuda")
    offset = torch.cumsum(length, 0) - length
    tube = torch.repeat_interleave(torch.arange(case["tubes"], device="cuda"), length)
    i = torch.arange(int(lengths.sum()), device="cuda") - offset[tube]
    side = ((i + 0.5) / length[tube] >= 0.5).long()
    rho, u, p = s[:, side, tube]
    return _euler1d(rho, u, p).contiguous(), lengths


def _dtype(case):
    return torch.float32 if case["prec"] == "f32" else torch.float64


# ------------------------------------------------------------- the library --
def prepare(case, seed):
    kind, prec = case["kind"], PREC[case["prec"]]
    if kind == "batch":
        U, lengths = _tubes64(case, seed)
        offsets = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
        ctx = B.Context(B.T7_EULER1D, int(offsets[-1]), 1.0 / case["nmax"], prec=prec,
                        bc=(B.T7_BC_ZERO_GRADIENT,) * 4)
        U = U.to(_dtype(case))
        return {"case": case, "ctx": ctx, "U": U, "W": torch.empty_like(U), "offsets": offsets, "dx": 1.0 / lengths}
    U = _state64(case, seed).to(_dtype(case)).contiguous()
    if kind == "gradient":
        dt = 0.25 / case["n"]  # CFL of about 0.55 for u = p = 1
        ctx = B.Context(B.T7_EULER1D, case["n"], _dx(case), prec=prec, bc=(B.T7_BC_PERIODIC,) * 4)
        g = torch.Generator(device="cuda").manual_seed(seed)
        v = torch.randn(U.shape, generator=g, dtype=torch.float64, device="cuda").to(U.dtype)
        return {"case": case, "ctx": ctx, "U": U.requires_grad_(), "v": v, "dt": dt}
    bc = (B.T7_BC_PERIODIC if _periodic(case) else B.T7_BC_ZERO_GRADIENT,) * 4
    two_d = case["system"] == "euler2d"
    ctx = B.Context(SYSTEM[case["system"]], case["n"], _dx(case), prec=prec, ny=case["ny"] if two_d else 1,
                    dy=1.0 / case["ny"] if two_d else 0.0, bc=bc)
    if kind == "host":
        H = torch.empty(U.shape, dtype=U.dtype, pin_memory=True)
        H.copy_(U)
        return {"case": case, "ctx": ctx, "H": H}
    if kind == "rhs":
        return {"case": case, "ctx": ctx, "U": U}
    return {"case": case, "ctx": ctx, "U": U, "W": torch.empty_like(U)}


def run(state):
    case, ctx = state["case"], state["ctx"]
    kind = case["kind"]
    if kind == "rhs":
        return ctx.euler_rhs(state["U"], want_masks=True)
    if kind == "batch":
        state["W"].copy_(state["U"])
        steps, t = ctx.batch_run(state["W"], state["offsets"], state["dx"], math.inf, 0.5, max_steps=case["steps"],
                                 group_warps=8)
        return state["W"], steps, t
    if kind == "gradient":
        out = A.CheckpointedRK3.apply(state["U"], ctx, state["dt"], case["steps"], case["every"])
        return out.detach(), torch.autograd.grad(out, state["U"], state["v"])[0]
    if kind == "host":
        ctx.run_host(state["H"], CFL[case["system"]], max_steps=case["steps"])
        return state["H"]
    state["W"].copy_(state["U"])
    steps, t = ctx.run(state["W"], CFL[case["system"]], t_end=case.get("t_end", math.inf), max_steps=case["steps"])
    return state["W"], steps, t


def work(case):
    size = 4 if case["prec"] == "f32" else 8
    if case["kind"] == "batch":
        cells = case["tubes"] * (case["nmin"] + case["nmax"]) // 2
        return {"bytes": 2 * 3 * cells * size, "flops": 3 * case["steps"] * cells * FLOPS["euler1d"]}
    if case["kind"] == "gradient":
        stages = 3 * case["steps"] * case["n"]
        return {"bytes": 4 * 3 * case["n"] * size, "flops": stages * (2 * FLOPS["euler1d"] + ADJOINT_FLOPS)}
    cells = case["n"] * case.get("ny", 1)
    m, flops = FIELDS[case["system"]], FLOPS[case["system"]] * cells
    if case["kind"] == "rhs":
        return {"bytes": 2 * m * cells * size + 2 * m * (cells + 1), "flops": flops}
    steps = case["steps"]
    if "t_end" in case:
        steps = min(steps, math.ceil(case["t_end"] / (CFL[case["system"]] * _dx(case))))
    return {"bytes": 2 * m * cells * size, "flops": 3 * steps * flops}


# --------------------------------------------------- the scheme in 64 bits --
_ROWS = [[-1 / 140, 5 / 84, -101 / 420, 319 / 420, 107 / 210, -19 / 210, 1 / 105],
         [0, 1 / 60, -2 / 15, 37 / 60, 37 / 60, -2 / 15, 1 / 60],
         [-1 / 60, 7 / 60, -23 / 60, 19 / 20, 11 / 30, -1 / 30, 0],
         [0, 0, -1 / 20, 9 / 20, 47 / 60, -13 / 60, 1 / 30],
         [0, 1 / 30, -13 / 60, 47 / 60, 9 / 20, -1 / 20, 0],
         [-1 / 20, 17 / 60, -43 / 60, 77 / 60, 1 / 5, 0, 0],
         [0, 0, 0, 1 / 4, 13 / 12, -5 / 12, 1 / 12],
         [0, 0, -1 / 12, 7 / 12, 7 / 12, -1 / 12, 0],
         [0, 1 / 12, -5 / 12, 13 / 12, 1 / 4, 0, 0],
         [-1 / 4, 13 / 12, -23 / 12, 25 / 12, 0, 0, 0],
         [0, 0, 0, 1 / 3, 5 / 6, -1 / 6, 0],
         [0, 0, -1 / 6, 5 / 6, 1 / 3, 0, 0],
         [0, 1 / 3, -7 / 6, 11 / 6, 0, 0, 0]]
# row of each Delta (first component in bit 4); the pattern (*,0,0,0,*) does not occur
_SELECT = [11, 11, 10, 6, 11, 11, 7, 3, 12, 12, 10, 6, 8, 8, 4, 1,
           11, 11, 10, 6, 11, 11, 7, 3, 9, 9, 10, 6, 5, 5, 2, 0]


def _kept(w, eps):
    """Cutoff bits (d0, d1, d2) of the five-point windows w."""
    b = [0.25 * (w[0] - 4 * w[1] + 3 * w[2]) ** 2 + 13 / 12 * (w[0] - 2 * w[1] + w[2]) ** 2,
         0.25 * (w[1] - w[3]) ** 2 + 13 / 12 * (w[1] - 2 * w[2] + w[3]) ** 2,
         0.25 * (3 * w[2] - 4 * w[3] + w[4]) ** 2 + 13 / 12 * (w[2] - 2 * w[3] + w[4]) ** 2]
    tau = (b[0] - b[2]).abs()
    y = [(1 + tau / (x + eps)) ** 6 for x in b]
    total = y[0] + y[1] + y[2]
    return [(x / total >= CT).long() for x in y]


def _reconstruct(q, eps):
    """Face values from the seven upwind-ordered taps q of every face, at the
    faces that have a neighbour on each side, and their Delta codes; the
    caller says which neighbour is upwind by the order of the faces."""
    with torch.no_grad():
        d = _kept([x.detach() for x in q[1:6]], eps)
        D = (d[0][..., :-2] << 4) | (d[0][..., 1:-1] << 3) | (d[1][..., 1:-1] << 2) | (d[2][..., 1:-1] << 1) \
            | d[2][..., 2:]
        row = torch.tensor(_SELECT, device=D.device)[D]
        table = torch.tensor(_ROWS, dtype=torch.float64, device=D.device)
    f = 0
    for t in range(7):
        f = f + table[:, t][row] * q[t][..., 1:-1]
    return f, D


def _physical(system, P):
    """Flux along the last axis and the quantities of the Roe average."""
    if system == "advection":
        return P, None
    if system == "burgers":
        return 0.5 * P * P, None
    rho, m, E = P[0], P[1], P[-1]
    u = m / rho
    kinetic = 0.5 * m * u
    if system == "euler2d":
        kinetic = kinetic + 0.5 * P[2] * P[2] / rho
    p = (GAMMA - 1.0) * (E - kinetic)
    flux = [m, m * u + p] + ([P[2] * u] if system == "euler2d" else []) + [u * (E + p)]
    prim = [u] + ([P[2] / rho] if system == "euler2d" else []) + [(E + p) / rho]
    return torch.stack(flux), (torch.sqrt(rho), torch.stack(prim))


def _frame(system, roe):
    """Left and right eigenvectors at every face (fields u-c, u, u+c; the shear
    field of 2D comes third), or None for the scalar laws."""
    if roe is None:
        return [[1.0]], [[1.0]]
    s, prim = roe
    sl, sr = s[..., 3:-4], s[..., 4:-3]
    avg = (sl * prim[..., 3:-4] + sr * prim[..., 4:-3]) / (sl + sr)
    u, H = avg[0], avg[-1]
    v = avg[1] if system == "euler2d" else 0.0
    k = 0.5 * (u * u + v * v)
    c2 = (GAMMA - 1.0) * (H - k)
    c = torch.sqrt(c2)
    b1 = (GAMMA - 1.0) / c2
    b2 = k * b1
    if system == "euler1d":
        return ([[0.5 * (b2 + u / c), -0.5 * (b1 * u + 1 / c), 0.5 * b1], [1 - b2, b1 * u, -b1],
                 [0.5 * (b2 - u / c), -0.5 * (b1 * u - 1 / c), 0.5 * b1]],
                [[1.0, 1.0, 1.0], [u - c, u, u + c], [H - u * c, k, H + u * c]])
    return ([[0.5 * (b2 + u / c), -0.5 * (b1 * u + 1 / c), -0.5 * b1 * v, 0.5 * b1],
             [1 - b2, b1 * u, b1 * v, -b1], [-v, 0.0, 1.0, 0.0],
             [0.5 * (b2 - u / c), -0.5 * (b1 * u - 1 / c), -0.5 * b1 * v, 0.5 * b1]],
            [[1.0, 1.0, 0.0, 1.0], [u - c, u, 0.0, u + c], [v, v, 1.0, v], [H - u * c, k, v, H + u * c]])


def _dot(row, parts):
    total = None
    for a, x in zip(row, parts):
        if isinstance(a, float):
            if a == 0.0:
                continue
            term = x if a == 1.0 else a * x
        else:
            term = a * x
        total = term if total is None else total + term
    return total


def _rhs_padded(system, P, alpha, dx, eps, codes=False):
    """L(U) along the last axis of P, padded by five cells per side; alpha and
    dx are numbers or values for each face and each cell.  Codes: Delta of
    both splits of every field at the faces of the inner cells."""
    m = P.shape[0]
    flux, roe = _physical(system, P)
    left, right = _frame(system, roe)
    S = P.shape[-1]
    a = alpha if not torch.is_tensor(alpha) or alpha.dim() == 0 else alpha
    plus, minus = 0.5 * (flux + a * P), 0.5 * (flux - a * P)
    shift = lambda X, t: X[..., t:S - 7 + t]  # the cell t - 3 places from each face's left cell
    f, D = [], [[], []]
    for k in range(m):
        up = [_dot(left[k], shift(plus, t)) for t in range(7)]
        fp, dp = _reconstruct(up, eps if not torch.is_tensor(eps) else eps[..., 3:-4])
        down = [_dot(left[k], shift(minus, 7 - t)).flip(-1) for t in range(7)]
        fm, dm = _reconstruct(down, eps if not torch.is_tensor(eps) else eps[..., 3:-4].flip(-1))
        f.append(fp + fm.flip(-1))
        D[0].append(dp)
        D[1].append(dm.flip(-1))
    inner = lambda x: x[..., 1:-1] if torch.is_tensor(x) else x
    F = torch.stack([_dot([inner(r) for r in right[k]], f) for k in range(m)])
    L = (F[..., :-1] - F[..., 1:]) / (dx if not torch.is_tensor(dx) else dx[..., 5:-5])
    return (L, torch.stack([torch.stack(x) for x in D])) if codes else L


def _pad(U, periodic, axis=-1):
    n = U.shape[axis]
    i = torch.arange(-5, n + 5, device=U.device)
    return U.index_select(axis, i % n if periodic else i.clamp(0, n - 1))


def _speed(system, U):
    """Characteristic speeds |u| + c of every cell (2D: both directions)."""
    if system == "advection":
        return [torch.ones_like(U[0])]
    if system == "burgers":
        return [U[0].abs()]
    u = [U[1] / U[0]] + ([U[2] / U[0]] if system == "euler2d" else [])
    p = (GAMMA - 1.0) * (U[-1] - 0.5 * U[0] * sum(x * x for x in u))
    c = torch.sqrt(GAMMA * p / U[0])
    return [x.abs() + c for x in u]


def _rhs(case, U, codes=False):
    system, dx = case.get("system", "euler1d"), _dx(case)
    alpha = [x.max() for x in _speed(system, U.detach())]
    periodic = _periodic(case)
    if system != "euler2d":
        return _rhs_padded(system, _pad(U, periodic), alpha[0], dx, dx ** 3, codes)
    dy = 1.0 / case["ny"]
    L = _rhs_padded(system, _pad(U, periodic), alpha[0], dx, dx ** 3)
    V = torch.stack([U[0], U[2], U[1], U[3]]).transpose(-1, -2)
    M = _rhs_padded(system, _pad(V, periodic), alpha[1], dy, dy ** 3).transpose(-1, -2)
    return L + torch.stack([M[0], M[2], M[1], M[3]])


def _rk3(U, dt, rhs):
    V = U + dt * rhs(U)
    V = 0.75 * U + 0.25 * (V + dt * rhs(V))
    return U / 3 + (V + dt * rhs(V)) * (2 / 3)


def _march(case, U):
    system, t, steps = case["system"], 0.0, 0
    t_end = case.get("t_end", math.inf)
    while steps < case["steps"] and t < t_end:
        alpha = [float(x.max()) for x in _speed(system, U)]
        if system == "euler2d":
            dt = CFL[system] / (alpha[0] / _dx(case) + alpha[1] * case["ny"])
        else:
            dt = CFL[system] * _dx(case) / alpha[0]
        dt = min(dt, t_end - t)
        U = _rk3(U, dt, lambda V: _rhs(case, V))
        t, steps = t + dt, steps + 1
    return U, steps, t


def _batch(case, U, lengths):
    """All tubes at once: each padded by its own end cells, one alpha and one
    step size for each."""
    tubes = case["tubes"]
    length = torch.tensor(lengths, device=U.device)
    padded = length + 10
    tube = torch.repeat_interleave(torch.arange(tubes, device=U.device), length)
    ptube = torch.repeat_interleave(torch.arange(tubes, device=U.device), padded)
    start, pstart = torch.cumsum(length, 0) - length, torch.cumsum(padded, 0) - padded
    i = torch.arange(int(padded.sum()), device=U.device) - pstart[ptube] - 5
    source = start[ptube] + torch.minimum(i.clamp(min=0), length[ptube] - 1)
    inner = torch.nonzero((i >= 0) & (i < length[ptube]))[:, 0] - 5
    dx = 1.0 / torch.tensor(lengths, dtype=torch.float64, device=U.device)
    pdx = dx[ptube]

    def alphas(V):
        return torch.zeros(tubes, dtype=torch.float64, device=U.device).scatter_reduce(
            0, tube, _speed("euler1d", V)[0], "amax")

    def rhs(V):
        return _rhs_padded("euler1d", V[:, source], alphas(V)[ptube], pdx, pdx ** 3)[:, inner]

    t = torch.zeros(tubes, dtype=torch.float64, device=U.device)
    for _ in range(case["steps"]):
        dt = 0.5 * dx / alphas(U)
        U = _rk3(U, dt[tube], rhs)
        t = t + dt
    return U, np.full(tubes, case["steps"], np.int32), t.cpu().numpy()


def exact(case, seed):
    """The pass's outputs from plain torch operations in 64 bits; None where
    that would take long."""
    kind = case["kind"]
    # every march step is some two thousand small launches here
    if kind in ("run", "batch", "host", "gradient"):
        cells = case["n"] * case.get("ny", 1) if kind != "batch" else case["tubes"] * case["nmax"] // 2
        if case["steps"] * (1 if kind == "gradient" else 0.25) > 130 and case.get("system") != "advection":
            return None
        if cells * case["steps"] > 70000000 * (6 if kind == "batch" else 1):
            return None
    with torch.set_grad_enabled(kind == "gradient"):
        if kind == "batch":
            U, lengths = _tubes64(case, seed)
            return _batch(case, U.to(_dtype(case)).double(), lengths)
        U = _state64(case, seed).to(_dtype(case)).double()
        if kind == "rhs":
            L, D = _rhs(case, U, codes=True)
            return L, (None if case["prec"] != "f64" else D.to(torch.uint8))
        if kind == "gradient":
            return _gradient(case, U, seed)
        U, steps, t = _march(case, U)
        return U.cpu() if kind == "host" else (U, steps, t)


def _gradient(case, U0, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    lam = torch.randn(U0.shape, generator=g, dtype=torch.float64, device="cuda").to(_dtype(case)).double()
    dt = 0.25 / case["n"]
    states = [U0.detach()]
    with torch.no_grad():
        for _ in range(case["steps"]):
            states.append(_rk3(states[-1], dt, lambda V: _rhs(case, V)))
    for U in reversed(states[:-1]):  # one step's graph at a time
        U = U.requires_grad_()
        lam = torch.autograd.grad(_rk3(U, dt, lambda V: _rhs(case, V)), U, lam)[0]
    return states[-1], lam
