"""The group size t7_batch_autotune keeps follows from the trial times it returns, as the
header states: the largest whose time is below 1.02 times the shortest."""
import numpy as np
import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", [B.T7_F64, B.T7_F32])
@pytest.mark.parametrize("ntubes,nmin,nmax", [(5, 12, 40), (64, 100, 2000), (700, 256, 700)])
def test_kept_group_follows_from_the_times(prec, ntubes, nmin, nmax):
    U, off, dx, _ = I.riemann_tube_batch(3, ntubes, nmin, nmax)
    c = B.Context(B.T7_EULER1D, U.shape[1], 1.0, prec=prec, bc=(1, 1, 0, 0))
    U = torch.tensor(U, dtype=c.dtype, device="cuda")
    for _ in range(4):
        group, ms = c.batch_autotune(U, off, dx, 0.5, trial_steps=4)
        close = ms < np.float32(1.02) * ms.min()
        assert group == max(g for g, ok in zip((1, 2, 4, 8), close) if ok), (group, ms)
    c.close()
