"""Correction and normal-equation solves in lockstep: what differs between right-hand sides.

Through the solvers that use them: a zero right-hand side beside others, shifts that
converge in very different numbers of iterations, the iteration budget, more right-hand
sides than one state holds, and sources whose sizes differ by many orders.  Solutions
are held to the requested true residual with the FP64 oracle.
"""
import numpy as np
import pytest

from oracle.dirac import gamma5
from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)


def test_shifts_of_very_different_size():
    qxd, ctx, op, _, _ = setup((4, 4, 6, 6), 1, PI, qhat=4, kappa=0.13)
    phi = workload.spinor(op.geom.V // 2, 5)
    sigma = [0.0, 1e-3, 8.4, 1e-6, 500.0, 0.3]
    x = np.empty((len(sigma),) + phi.shape, dtype=np.complex128)
    info = ctx.solve_multishift(0, sigma, phi, x, tol=1e-11, inner=qxd.FP32)
    Dinv = op.Doo_inv()
    for s, xj in zip(sigma, x):
        y = op.Dhat(gamma5(op.Dhat(xj, Dinv)), Dinv)
        r = phi - gamma5(y) - s * xj
        assert np.linalg.norm(r) <= 1.01e-11 * np.linalg.norm(phi)
    # too small a budget is reported, not exceeded by more than a chunk of eight iterations per shift
    low = info.iters // 2
    short = ctx.solve_multishift(0, sigma, phi, x, tol=1e-11, inner=qxd.FP32, nmx=low, check=False)
    assert short.status == 2 and short.iters <= low + 8 * len(sigma)
    ctx.close()


@pytest.mark.parametrize("nrhs", [3, 34])
def test_normal_equations_of_several_right_hand_sides(nrhs):
    # smooth links at a negative bare mass: restarted GCR stalls, CG on the normal equations takes over
    qxd, ctx, op, _, _ = setup((8, 8, 8, 8), 0, PI, kappa=0.136377, stout=5)
    eta = workload.spinor(op.geom.V, 7, nrhs=nrhs)
    eta[1] *= 1e-8
    eta[2] = 0.0
    psi = np.empty_like(eta)
    ctx.solve(0, eta, psi, nkv=2, inner=qxd.FP32, nrhs=nrhs, tol=1e-10)
    for j in (0, 1, nrhs - 1):
        if j != 2:
            assert np.linalg.norm(eta[j] - op.apply(psi[j])) <= 1e-10 * np.linalg.norm(eta[j])
    assert not psi[2].any()
    bad = eta.copy()
    bad[0, 3] = np.nan
    with pytest.raises(qxd.QxdError):
        ctx.solve(0, bad, psi, nkv=2, inner=qxd.FP32, nrhs=nrhs, tol=1e-10)
    ctx.close()
