"""Site-diagonal terms on lattices whose clover leaves do not fit the workspace at once.

The leaves are then formed slab by slab in x0, each with the slice before it.  Checked
through D at sampled sites (the first and last slices and the slab borders among them)
against the FP64 oracle, to the parity bar of FP64 operator applications (1e-13).
"""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import need_gpu, relerr, setup

pytestmark = pytest.mark.gpu


# a slab holds 512 MB / (1776 bytes x stored sites of a slice) slices: 36 here, 75 with C*
@pytest.mark.parametrize("L,cstar,tbc", [((40, 20, 20, 20), 0, "periodic"), ((40, 20, 20, 20), 0, "open"),
                                         ((78, 10, 20, 20), 1, "periodic")])
def test_site_diagonal_terms_in_slabs(L, cstar, tbc):
    need_gpu()
    theta = (0.0 if tbc == "open" else np.pi, 0.0, 0.0, 0.0)
    qxd, ctx, op, _, _ = setup(L, cstar, theta, qhat=4, kappa=0.13, device="cuda", tbc=tbc, cF=1.1)
    psi = workload.spinor(op.geom.V, 5)
    out = np.empty_like(psi)
    ctx.apply_Dw(0, qxd.FP64, psi, out)
    ctx.close()
    V = op.geom.V
    slice_ = V // L[0]
    rng = np.random.default_rng(1)
    x0 = [0, 1, 34, 35, 36, 37, L[0] - 4, L[0] - 2, L[0] - 1]
    sites = np.unique(np.concatenate([rng.integers(0, V, 200)] + [x * slice_ + rng.integers(0, slice_, 40) for x in x0]))
    ref = op.apply(psi, sites)
    for x in x0:
        at = sites // slice_ == x
        assert relerr(out[sites[at]], ref[at]) <= 1e-13
    assert relerr(out[sites], ref) <= 1e-13
