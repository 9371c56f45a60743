"""The iteration limit of solves in lockstep: one slow right-hand side among others that need
nothing, and shifts that share what is left of the limit."""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)


@pytest.mark.parametrize("nrhs,nmx", [(4, 21), (34, 30)])
def test_right_hand_sides_that_stop_leave_nothing_to_the_others(nrhs, nmx):
    # restarted GCR stalls here and CG on the normal equations takes over; an iteration of it is
    # two applications of Dhat, and each right-hand side has the limit for itself
    qxd, ctx, op, _, _ = setup((8, 8, 8, 8), 0, PI, kappa=0.136377, stout=5)
    eta = np.zeros((nrhs, op.geom.V, 4, 3), dtype=complex)
    eta[1] = workload.spinor(op.geom.V, 7)
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=2, inner=qxd.FP32, nrhs=nrhs, tol=1e-10, nmx=nmx, check=False)
    assert info.status == 2 and nmx <= info.iters <= 2 * nmx
    ctx.close()


def test_shifts_share_exactly_what_is_left():
    qxd, ctx, op, _, _ = setup((4, 4, 6, 6), 1, PI, qhat=4, kappa=0.13)
    phi = workload.spinor(op.geom.V // 2, 5)
    sigma = [0.0, 1e-3, 8.4, 1e-6, 500.0, 0.3]
    x = np.empty((len(sigma),) + phi.shape, dtype=np.complex128)
    full = ctx.solve_multishift(0, sigma, phi, x, tol=1e-11, inner=qxd.FP32).iters
    for nmx in range(full // 3, full, 3):  # some of these end in the middle of a step of all shifts
        info = ctx.solve_multishift(0, sigma, phi, x, tol=1e-11, inner=qxd.FP32, nmx=nmx, check=False)
        assert info.status == 2 and info.iters <= nmx, nmx
    again = ctx.solve_multishift(0, sigma, phi, x, tol=1e-11, inner=qxd.FP32, nmx=full)
    assert again.iters == full
    ctx.close()
