"""The last stage of a host-array run in one, two, several and eight parts (parts
of at least 2 MB): the same values, bit for bit, as the device run."""
import numpy as np
import pytest

from paper_1808_00037_gb300 import binding as B
from paper_1808_00037_gb300 import inputs as I

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec,dtype", [(B.T7_F64, torch.float64), (B.T7_F32, torch.float32),
                                        (B.T7_MIXED, torch.float64)])
@pytest.mark.parametrize("mb", [0.01, 1.9, 4.01, 11.3, 17.0])
def test_parts_equal_device_run(prec, dtype, mb):
    cells = int(mb * 2**20) // (3 * (8 if dtype == torch.float64 else 4)) | 1
    U, dx = I.shu_osher(1600, tiles=cells // 1600 + 1)
    U = np.ascontiguousarray(U[:, :cells])
    c = B.Context(B.T7_EULER1D, cells, dx, prec=prec, bc=(1, 1, 0, 0))
    Ud = torch.tensor(U, dtype=dtype, device="cuda")
    sd, td = c.run(Ud, 0.5, max_steps=2)
    Uh = torch.tensor(U, dtype=dtype).pin_memory()
    sh, th = c.run_host(Uh, 0.5, max_steps=2)
    assert (sd, td) == (sh, th)
    assert torch.equal(Ud.cpu(), Uh)
