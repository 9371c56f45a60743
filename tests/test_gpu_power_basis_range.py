"""Unpreconditioned FP32 inner solves at the ends of the power basis: sources far from 1 in
size."""
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
