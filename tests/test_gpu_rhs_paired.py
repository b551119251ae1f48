"""One-launch right-hand sides, steps and recorded steps on FP32 tiles with paired faces,
at the ends of that form's range and with one, two and several tiles a warp, against
launches of single stages (which a capture into a CUDA graph takes): the same bits, in
values, codes, alphas and stage states."""
import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


# 61 cells a tile, 8 tiles a block, 304 blocks: two tiles a warp from 148,353 cells on
@pytest.mark.parametrize("system,n", [
    ("euler", 29 * 1216 + 1), ("euler", 61 * 8 * 152), ("euler", 61 * 8 * 152 + 1), ("euler", 148352),
    ("euler", 148353), ("euler", 400_009), ("euler", 1 << 20), ("euler", (1 << 20) + 1),
    ("burgers", 29 * 304 + 1), ("burgers", 29 * 1064), ("burgers", 29 * 1064 + 1)])
def test_one_launch_equals_stage_launches(system, n):
    if system == "euler":
        U, dx = I.shu_osher(n)
        sys_, bc = B.T7_EULER1D, 1
    else:
        U, dx, _ = I.burgers_sine(n)
        sys_, bc = B.T7_BURGERS, 0
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        c = B.Context(sys_, n, dx, prec=B.T7_F32, bc=(bc,) * 4, stream=s)
        A = torch.tensor(U, dtype=c.dtype, device="cuda")
        dt = c.cfl_dt(A, 0.4)
        record = system == "euler"
        tapes = [torch.zeros(c.tape_bytes() if record else 1, dtype=torch.uint8, device="cuda") for _ in range(2)]
        masks = [torch.zeros((2, c.m, n + 1), dtype=torch.uint8, device="cuda") for _ in range(2)]
        outs = [[torch.zeros_like(A) for _ in range(3)] for _ in range(2)]

        def calls(k):
            c._check(c.lib.t7_euler_rhs(c.h, A.data_ptr(), outs[k][0].data_ptr(), masks[k].data_ptr()), "t7_euler_rhs")
            outs[k][1].copy_(A)
            c.rk3_step(outs[k][1], dt)
            if record:
                c.rk3_step_record(A, outs[k][2], dt, tapes[k])

        calls(0)
        c.sync()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=s):
            calls(1)
        g.replay()
        c.sync()
        assert all(torch.equal(a, b) for a, b in zip(*outs))
        assert torch.equal(*masks) and torch.equal(*tapes)
        c.close()
