"""The residual norm of preconditioned GCR: summed where the recursion loses digits, and only there,
because the host waits for it."""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu


def test_norms_are_not_summed_in_every_step():
    qxd, ctx, op, _, _ = setup((4, 4, 4, 4), 0, (np.pi, 0.0, 0.0, 0.0), kappa=0.126)
    W = np.zeros((1, 1, 9, 4, 4), dtype=np.complex64)
    W[0, 0, 0] = 0.252 * np.eye(4)  # one layer: 2 kappa times the residual
    ctx.set_precond_weights(0, W, 1, 1, qxd.FP32)
    eta = workload.spinor(op.geom.V, 5)
    psi = np.empty_like(eta)
    ctx.profile(1)
    info = ctx.solve(0, eta, psi, nkv=8, inner=qxd.FP32, precond=qxd.PRECOND_LEARNED, tol=1e-10)
    n = {p["name"]: p["launches"] for p in ctx.profile_entries()}
    ctx.profile(0)
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-10 * np.linalg.norm(eta)
    # seven of eight steps orthogonalise in such a pass, restarts take one; a step reduces |r|^2 by
    # about two to eight here, so that one in three at most falls a hundredfold below the last sum
    assert n["multi_axpy_norm"] < 1.5 * info.iters
    ctx.close()
