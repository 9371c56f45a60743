"""Unpreconditioned FP32 inner solves at the ends of the power basis: sources far from 1 in
size, and the tolerance of the inner solves."""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nkv,exponent", [(8, 54), (12, 52), (16, 50)])
def test_large_sources(nkv, exponent):
    # a power of two scales every number of the solve exactly: same iterations, same bits
    qxd, ctx, op, _, _ = setup((4, 4, 6, 8), 0, (np.pi, 0.0, 0.0, 0.0), kappa=0.134, stout=5)
    eta = workload.spinor(op.geom.V, 5)
    psi, big = np.empty_like(eta), np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-10 * np.linalg.norm(eta)
    scaled = ctx.solve(0, eta * 2.0 ** exponent, big, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    assert scaled.iters == info.iters
    assert np.array_equal(big, psi * 2.0 ** exponent)
    ctx.close()


@pytest.mark.parametrize("L,kappa,stout,nkv", [((4, 4, 6, 8), 0.134, 5, 8), ((4, 4, 6, 8), 0.134, 5, 12),
                                               ((4, 4, 6, 8), 0.134, 5, 16), ((8, 8, 8, 8), 0.126, 0, 12),
                                               ((8, 8, 8, 8), 0.126, 0, 16)])
def test_inner_solves_reach_their_tolerance(L, kappa, stout, nkv):
    # two inner solves to 1e-5 of an even-odd source that is smaller than the source reach 1e-10
    qxd, ctx, op, _, _ = setup(L, 0, (np.pi, 0.0, 0.0, 0.0), kappa=kappa, stout=stout)
    eta = workload.spinor(op.geom.V, 5)
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    ev, od = op.even_sites(), op.odd_sites()
    b = eta[ev] - op.Deo(np.einsum("nab,nb->na", op.Doo_inv(), eta[od].reshape(-1, 12)).reshape(-1, 4, 3))
    assert np.linalg.norm(b) < np.linalg.norm(eta)
    assert info.restarts == 1
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-10 * np.linalg.norm(eta)
    ctx.close()
