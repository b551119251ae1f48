"""The adjoint on domains of two cells to a few tiles (25 cells each): cells near the ends,
their ghosts' shares and domains shorter than a stencil.  The whole transposed
Jacobian-vector product against the Jacobian that the oracle's tangent-linear mode gives
column by column, with the selection the forward kernels take.

An entry of J is a sum of some 100 products; the frame's cancellations enlarge their
rounding by less than 100 for these states.  So an entry of J^T v is within
1e4 2^-53 = 1.2e-12 (FP32 6e-4) of |J|^T |v|, and a step's three stages, each linear in
the one before, within a few times that.  (A single cell's right-hand side is constant:
its J is zero by cancellation, and no such bound exists.)"""
import numpy as np
import pytest

import oracle
from paper_1808_00037_gb300 import binding as B

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

SIZES = [2, 3, 4, 5, 7, 8, 9, 16, 17, 18, 25, 26, 42, 43, 67, 92, 93, 121]
TOL = {B.T7_F64: 1.2e-12, B.T7_F32: 6e-4}


def state(n, seed, prec):
    rng = np.random.default_rng(seed)
    rho, u, p = 1 + 0.4 * rng.random(n), 0.3 * rng.normal(size=n), 1 + 0.4 * rng.random(n)
    if n > 8:
        p[n // 2:] += 2.0  # a jump
    U = np.stack([rho, rho * u, p / 0.4 + 0.5 * rho * u * u])
    if prec == B.T7_F32:
        U = U.astype(np.float32).astype(np.float64)
    return U, 0.1


@pytest.mark.parametrize("prec", [B.T7_F64, B.T7_F32])
@pytest.mark.parametrize("bc", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n", SIZES)
def test_rhs_adjoint_is_the_transposed_jacobian(n, bc, prec):
    U, dx = state(n, 100 + n, prec)
    c = B.Context(B.T7_EULER1D, n, dx, prec=prec, bc=(bc[0], bc[1], 0, 0))
    Ud = torch.tensor(U, dtype=c.dtype, device="cuda")
    masks = c.euler_rhs(Ud, want_masks=True)[1].cpu().numpy()
    v = torch.tensor(np.random.default_rng(n).normal(size=U.shape), dtype=c.dtype, device="cuda")
    out = c.euler_rhs_adjoint(Ud, v)
    c.sync()
    alpha = oracle.rhs_1d(oracle.SYS_EULER1D, U, dx, bc=bc)[1]
    J = np.empty((3 * n, 3 * n))
    for k in range(3 * n):
        e = np.zeros(3 * n)
        e[k] = 1.0
        J[:, k] = oracle.rhs_1d_tl(oracle.SYS_EULER1D, U, e.reshape(3, n), dx, alpha, masks, bc=bc)[1].ravel()
    v = v.double().cpu().numpy().ravel()
    d = np.abs(out.double().cpu().numpy().ravel() - J.T @ v)
    assert np.all(d <= TOL[prec] * (np.abs(J).T @ np.abs(v)))
    c.close()


@pytest.mark.parametrize("bc", [(0, 0), (1, 1)])
@pytest.mark.parametrize("n", SIZES)
def test_step_adjoints_are_the_transposed_jacobian(n, bc):
    U, dx = state(n, 200 + n, B.T7_F64)
    c = B.Context(B.T7_EULER1D, n, dx, bc=(bc[0], bc[1], 0, 0))
    Ud = torch.tensor(U, device="cuda")
    dt = c.cfl_dt(Ud, 0.4)
    lam = torch.tensor(np.random.default_rng(n).normal(size=U.shape), device="cuda")
    tape = torch.empty(c.tape_bytes(), dtype=torch.uint8, device="cuda")
    c.rk3_step_record(Ud, torch.empty_like(Ud), dt, tape)
    got = [c.rk3_step_adjoint(Ud, dt, lam.clone()), c.rk3_step_adjoint_recorded(Ud, tape, dt, lam.clone())]
    c.sync()
    J = np.empty((3 * n, 3 * n))
    for k in range(3 * n):
        e = np.zeros(3 * n)
        e[k] = 1.0
        J[:, k] = oracle.rk3_step_1d_tl(oracle.SYS_EULER1D, U, e.reshape(3, n), dx, dt, bc=bc)[1].ravel()
    v = lam.cpu().numpy().ravel()
    for g in got:
        d = np.abs(g.cpu().numpy().ravel() - J.T @ v)
        assert np.all(d <= 10 * TOL[B.T7_F64] * (np.abs(J).T @ np.abs(v)))
    c.close()
