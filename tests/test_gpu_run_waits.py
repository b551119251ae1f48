"""The waits between the blocks of one-launch runs, steps and right-hand sides: a wait
that runs out (in the checked build t7_probe_run_waits makes one block give up at its
first) returns T7_ETIMEOUT, ends the run's later launches at once, and leaves the
context usable; and the exchange tags restart over cleared slots.  Sizes whose launch is a grid of waiting
blocks: FP64 with a tile per block, FP32 and mixed with a tile per warp, FP32 with
paired faces."""
import ctypes
import math

import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import build
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

FORMS = [(B.T7_F64, 1000), (B.T7_F32, 5000), (B.T7_F32, 40000), (B.T7_MIXED, 5000)]


@pytest.fixture
def checked(monkeypatch):
    """Contexts of the checked build, whose waits can be made to run out."""
    monkeypatch.setattr(B, "_lib", B.load(build.build(checked=True)))


def context(prec, n):
    U, dx = I.shu_osher(n)
    c = B.Context(B.T7_EULER1D, n, dx, prec=prec, bc=(1, 1, 0, 0))
    return c, torch.tensor(U, dtype=c.dtype, device="cuda")


def DT(c):
    return 0.08 * c.grid.dx  # CFL 0.4: the largest wave speed is 4.57


def rhs(c, U):
    return c.euler_rhs(U)[0]


def step(c, U):
    return c.rk3_step(U.clone(), DT(c))


def record(c, U):
    tape = torch.empty(c.tape_bytes(), dtype=torch.uint8, device="cuda")
    return c.rk3_step_record(U, torch.empty_like(U), DT(c), tape)


def run(c, U):
    A = U.clone()
    c.run(A, 0.5, max_steps=130)
    return A


def run_host(c, U):
    H = U.cpu()
    c.run_host(H, 0.5, max_steps=130)
    return H


@pytest.mark.parametrize("call", [rhs, step, record, run, run_host], ids=lambda f: f.__name__)
@pytest.mark.parametrize("prec,n", FORMS)
@pytest.mark.parametrize("block", [0, 1, 19])
def test_wait_that_runs_out(checked, prec, n, call, block):
    if prec == B.T7_MIXED and call not in (run, run_host):
        pytest.skip("mixed precision has the one-launch run only")
    c, U = context(prec, n)
    c.probe_run_waits(block, polls=1 << 12)
    with pytest.raises(B.T7Error) as e:
        call(c, U)
        c.sync()
    assert e.value.status == B.T7_ETIMEOUT
    got = call(c, U)
    c.sync()
    fresh, U = context(prec, n)
    want = call(fresh, U)
    fresh.sync()
    assert torch.equal(got, want)
    c.close()
    fresh.close()


@pytest.mark.parametrize("prec,n", FORMS)
def test_run_ends_where_a_wait_ran_out(checked, prec, n):
    """The launches queued after the one whose wait ran out advance nothing."""
    c, U = context(prec, n)
    c.probe_run_waits(1, polls=1 << 12)
    steps, t = ctypes.c_int(-1), ctypes.c_double(-1.0)
    st = c.lib.t7_run(c.h, U.data_ptr(), 0.5, math.inf, 192, ctypes.byref(steps), ctypes.byref(t))
    c.close()
    assert (st, steps.value, t.value) == (B.T7_ETIMEOUT, 0, 0.0)


@pytest.mark.parametrize("prec,n", FORMS)
@pytest.mark.parametrize("left", [0, 192, 193, 300])
def test_tags_restart(prec, n, left):
    c, U = context(prec, n)
    c.probe_run_waits(tag=(1 << 32) - 1 - left)
    got = run(c, U)
    for bad in (dict(tag=1), dict(block=1)):  # below the present tag; release build
        with pytest.raises(B.T7Error):
            c.probe_run_waits(**bad)
    fresh, U = context(prec, n)
    assert torch.equal(got, run(fresh, U))
    if prec != B.T7_MIXED:
        assert torch.equal(rhs(c, U), rhs(fresh, U))
        c.sync()
        fresh.sync()
