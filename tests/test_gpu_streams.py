"""Small 1D problems on several streams at once: one-launch grids that would not fit the
chip beside the others' give way to launches of single stages (they would run one after
another), and the results stay the same bit for bit.  Which form a call takes shows in
the checked build, where the waits of a one-launch form can be made to run out
(t7_probe_run_waits) and stage launches have none."""
import gc
import threading
import time

import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import build
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def context(prec, n, stream):
    U, dx = I.shu_osher(n)
    with torch.cuda.stream(stream):
        c = B.Context(B.T7_EULER1D, n, dx, prec=prec, bc=(1, 1, 0, 0), stream=stream)
        U = torch.tensor(U, dtype=c.dtype, device="cuda")
    stream.synchronize()
    return c, U


def waits(c, call):
    """Whether the call is a one-launch form (its wait is made to run out)."""
    c.probe_run_waits(1, polls=1 << 12)
    try:
        call()
        c.sync()
    except B.T7Error as e:
        assert e.status == B.T7_ETIMEOUT
        return True
    return False


@pytest.fixture
def checked(monkeypatch):
    gc.collect()  # no context of an earlier test is left on a stream of its own
    monkeypatch.setattr(B, "_lib", B.load(build.build(checked=True)))


# (the grids: 22 and 304 blocks of 304 in FP32 / FP64 at the sizes' ends)
@pytest.mark.parametrize("prec,n,rhs_several,step_several", [
    (B.T7_F32, 5000, True, True), (B.T7_F32, 50000, True, False), (B.T7_F32, 100003, False, False),
    (B.T7_F64, 1600, True, True), (B.T7_F64, 8000, False, False)])
def test_calls_of_contexts_on_several_streams(checked, prec, n, rhs_several, step_several):
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    c, U = context(prec, n, s1)
    other, _ = context(prec, 100, s1)
    dt = 0.01 * c.grid.dx

    def forms():
        return (waits(c, lambda: c.euler_rhs(U, out=torch.empty_like(U))),
                waits(c, lambda: c.rk3_step(U.clone(), dt)))

    with torch.cuda.stream(s1):
        assert forms() == (True, True)
        other.set_stream(s2)
        assert forms() == (rhs_several, step_several)
        other.set_stream(s1)
        assert forms() == (True, True)
        third, _ = context(prec, 100, s2)
        assert forms() == (rhs_several, step_several)
        third.close()
        assert forms() == (True, True)
    c.close()
    other.close()


def test_run_beside_a_run_in_progress(checked):
    s1, s2 = torch.cuda.Stream(), torch.cuda.Stream()
    long, V = context(B.T7_F64, 1_000_003, s1)
    # 22, 87 and 205 blocks of 304: beside one other run, and alone with a context on another stream
    cases = [(context(B.T7_F32, n, s2), beside) for n, beside in ((5000, True), (20000, True), (100003, False))]
    done = []

    def march():
        long.run(V, 0.2, max_steps=1500)
        done.append(True)

    def forms():
        with torch.cuda.stream(s2):  # (the copies are made on the runs' stream)
            return [waits(c, lambda: c.run(U.clone(), 0.2, max_steps=3)) for (c, U), _ in cases]

    th = threading.Thread(target=march)
    th.start()
    time.sleep(0.3)
    got = forms()
    assert not done  # the long run was in progress all the while
    th.join()
    assert got == forms() == [beside for _, beside in cases]
    long.close()
    assert all(forms())


@pytest.mark.parametrize("prec,n", [(B.T7_F64, 4000), (B.T7_F64, 9001), (B.T7_F32, 20000), (B.T7_F32, 100003),
                                    (B.T7_MIXED, 30000)])
def test_runs_at_once_equal_runs_alone(prec, n):
    jobs = [context(prec, n, torch.cuda.Stream()) for _ in range(6)]
    steps = [130 + 9 * k for k in range(6)]
    out = {}

    def march(k):
        c, U = jobs[k]
        with torch.cuda.stream(c.stream):
            A = U.clone()
            out[k] = c.run(A, 0.4, max_steps=steps[k]), A

    threads = [threading.Thread(target=march, args=(k,)) for k in range(6)]
    for th in threads:
        th.start()
    for th in threads:
        th.join()
    at_once = dict(out)
    for k in range(6):
        march(k)
        assert out[k][0] == at_once[k][0] and torch.equal(out[k][1], at_once[k][1]), k
