"""Batches of fewer tubes than the GPU holds CTAs, whose tubes each run on a
cluster of 2, 4 or 8 CTAs (group_warps = 8), against groups of four warps
(group_warps = 4): every value, step count and time is the same bit for bit.
Lengths around a tile (29 cells), tubes with fewer tiles than the cluster has
warps, and more tubes than clusters fit at once."""
import numpy as np
import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [B.T7_F64, B.T7_F32])
@pytest.mark.parametrize("ntubes,nmin,nmax,t_end,max_steps", [
    (1, 2500, 2500, np.inf, 7),   # one tube, eight CTAs
    (3, 232, 1900, 0.01, 1 << 30),  # uneven step counts, to a common time
    (20, 12, 2000, np.inf, 5),    # tubes shorter than a tile beside long ones
    (40, 260, 700, np.inf, 0),    # no step at all
    (60, 29, 1200, np.inf, 4),
    (140, 233, 500, np.inf, 3),
    (290, 240, 300, np.inf, 3),
])
def test_cluster_tubes_equal_group_tubes(prec, ntubes, nmin, nmax, t_end, max_steps):
    U, off, dx, _ = I.riemann_tube_batch(17 + ntubes, ntubes, nmin, nmax)
    c = B.Context(B.T7_EULER1D, U.shape[1], 1.0, prec=prec, bc=(1, 1, 0, 0))
    dt = torch.float64 if prec == B.T7_F64 else torch.float32
    out = []
    for group in (4, 8):
        Ug = torch.tensor(U, dtype=dt, device="cuda")
        steps, t = c.batch_run(Ug, off, dx, t_end, 0.5, max_steps=max_steps, group_warps=group)
        out.append((Ug.cpu().numpy(), steps, t))
    (U4, s4, t4), (U8, s8, t8) = out
    assert np.array_equal(s8, s4) and np.array_equal(t8, t4)
    assert np.array_equal(U8, U4)
    assert s4.min() >= 1 or max_steps == 0
