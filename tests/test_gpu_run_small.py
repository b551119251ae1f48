"""t7_run on small 1D domains, which marches whole steps in one launch: sizes at
the edges of its tiles, CTAs, clusters and of the one-tile-per-CTA FP64 form."""
import math

import numpy as np
import pytest

import oracle
from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import inputs as I

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# cells: one; a tile (29) and beside; 8, 16, 64 and 128 tiles and one cell more; and past 152, 304, 912, 1064 and
# 1216 tiles, where the form changes
SIZES = [1, 28, 29, 30, 232, 233, 464, 465, 1856, 1857, 3712, 3713, 29 * 152 + 1, 29 * 304 + 1, 29 * 912 + 1,
         29 * 1064 + 1, 29 * 1216 + 1]
SYSTEMS = {"advection": (B.T7_SCALAR_ADVECTION, 0.2, 0), "burgers": (B.T7_BURGERS, 0.5, 0),
           "euler": (B.T7_EULER1D, 0.5, 1)}


def state(system, n):
    if system == "euler":
        return I.shu_osher(n)
    U, dx, _ = I.burgers_sine(n) if system == "burgers" else I.advection_sine(n)
    return U, dx


@pytest.mark.parametrize("scheme", [B.T7_TENO7EXT, B.T7_TENO5])
@pytest.mark.parametrize("system", sorted(SYSTEMS))
@pytest.mark.parametrize("n", SIZES)
def test_run_equals_stage_launches(system, n, scheme):
    """The march equals the stage-by-stage launches bit for bit: in every precision
    those of t7_run_host (whose last chunk of steps is never one launch), and in
    FP64 t7_cfl_dt and t7_rk3_step called step by step, the last step clipped."""
    sys_, cfl, bc = SYSTEMS[system]
    U, dx = state(system, n)
    for prec in (B.T7_F64, B.T7_F32, B.T7_MIXED):
        ctx = B.Context(sys_, n, dx, prec=prec, bc=(bc,) * 4, scheme=scheme)
        A = torch.tensor(U, dtype=ctx.dtype, device="cuda")
        H, S, t = A.cpu(), A.clone(), 0.0
        assert ctx.run(A, cfl, max_steps=3) == ctx.run_host(H, cfl, max_steps=3)
        assert torch.equal(A.cpu(), H), prec
        if prec != B.T7_F64:
            continue
        A = S.clone()
        for _ in range(3):
            dt = ctx.cfl_dt(S, cfl)
            ctx.rk3_step(S, dt)
            t += dt
        ctx.sync()
        assert ctx.run(A, cfl, t_end=t) == (3, t) and torch.equal(A, S)
        ctx.close()


@pytest.mark.parametrize("n", [29 * 9 + 3, 29 * 152, 29 * 160])
def test_long_run_matches_oracle(n):
    """Chunk after chunk of the march (FP64 Euler) is the oracle's run, bit for bit."""
    U, dx = I.shu_osher(n)
    Uo, so, to, _ = oracle.run_1d(oracle.SYS_EULER1D, U, dx, t_end=math.inf, cfl=0.5, bc=(1, 1), max_steps=70)
    ctx = B.Context(B.T7_EULER1D, n, dx, bc=(1, 1, 0, 0))
    A = torch.tensor(U, device="cuda")
    steps, t = ctx.run(A, 0.5, max_steps=70)
    assert (steps, t) == (so, to) and np.array_equal(A.cpu().numpy(), Uo)
    ctx.close()


def test_runs_on_several_streams_and_threads():
    """Contexts marching at once on their own streams and threads give what each gives alone."""
    import threading

    jobs = [("euler", 1600, B.T7_F64), ("euler", 3000, B.T7_F32), ("advection", 200, B.T7_F64),
            ("burgers", 2000, B.T7_F32)]
    want, got = {}, {}

    def march(k, out):
        system, n, prec = jobs[k]
        sys_, cfl, bc = SYSTEMS[system]
        U, dx = state(system, n)
        s = torch.cuda.Stream()
        with torch.cuda.stream(s):
            ctx = B.Context(sys_, n, dx, prec=prec, bc=(bc,) * 4, stream=s)
            A = torch.tensor(U, dtype=ctx.dtype, device="cuda")
            s.synchronize()
            ctx.run(A, cfl, max_steps=150)
        out[k] = A.cpu()
        ctx.close()

    for k in range(len(jobs)):
        march(k, want)
    threads = [threading.Thread(target=march, args=(k, got)) for k in range(len(jobs))]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    for k in range(len(jobs)):
        assert torch.equal(want[k], got[k]), jobs[k]


@pytest.mark.parametrize("prec", [B.T7_F64, B.T7_F32])
@pytest.mark.parametrize("system", sorted(SYSTEMS))
@pytest.mark.parametrize("n", [5, 29 * 16 + 7, 29 * 304, 29 * 304 + 1, 29 * 1216 + 1])
def test_rhs_and_step_under_capture(system, n, prec):
    """t7_euler_rhs and t7_rk3_step captured into a CUDA graph (where they are
    launches of single stages) and replayed equal the plain calls, bit for bit."""
    sys_, cfl, bc = SYSTEMS[system]
    U, dx = state(system, n)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        ctx = B.Context(sys_, n, dx, prec=prec, bc=(bc,) * 4, stream=s)
        A = torch.tensor(U, dtype=ctx.dtype, device="cuda")
        S, out, out_s = A.clone(), torch.empty_like(A), torch.empty_like(A)
        dt = ctx.cfl_dt(A, cfl)
        s.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            ctx.euler_rhs(A, out=out)
            ctx.rk3_step(A, dt)
        for _ in range(3):
            g.replay()
            ctx.euler_rhs(S, out=out_s)
            ctx.rk3_step(S, dt)
            ctx.sync()
            assert torch.equal(out, out_s) and torch.equal(A, S)
        ctx.close()
