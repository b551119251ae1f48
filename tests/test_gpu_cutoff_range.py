"""FP64 stencil codes of values up to and beyond what FP32 squares hold: the smoothness
measures' reciprocals are FP32 ones, whose results vanish above 2^126.  The
reconstruction's codes and values, and the right-hand side's of a scalar law, are the
oracle's bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1808_00037_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def values(scale, n=20000):
    rng = np.random.default_rng(4)
    v = np.repeat(rng.normal(size=n // 5 + 1), 5)[:n] + rng.normal(size=n) * 10.0 ** rng.integers(-6, 0, size=n)
    return v * scale


@pytest.mark.parametrize("scale", [1e-20, 1e-18, 1.0, 1e17, 1e18, 3e18, 6e18, 1e19, 1e20])
def test_codes_of_large_and_small_values(scale):
    v = values(scale)
    n = v.size - 8
    c = B.Context(B.T7_SCALAR_ADVECTION, n, 0.01)
    for sign in (1, -1):
        fo, d3o, D5o = oracle.teno7_reconstruct(v, sign, 1e-6)
        fg, d3g, D5g = c.teno7_reconstruct(torch.tensor(v, device="cuda"), sign, 1e-6, want_bits=True)
        c.sync()
        assert np.array_equal(d3g.cpu().numpy(), d3o) and np.array_equal(D5g.cpu().numpy(), D5o)
        assert np.array_equal(fg.cpu().numpy(), fo)
    ro, _, mo = oracle.rhs_1d(oracle.SYS_ADVECTION, v[None, :n], 0.01, want_masks=True)
    rg, mg = c.euler_rhs(torch.tensor(np.ascontiguousarray(v[None, :n]), device="cuda"), want_masks=True)
    c.sync()
    assert np.array_equal(mg.cpu().numpy(), mo) and np.array_equal(rg.cpu().numpy(), ro)
    c.close()
