"""Network layers and weight gradients at the shapes where their kernels differ.

Channel counts on both sides of the kernels' groups (1, 2, 4, 8 and remainders), one to
three layers (first and last layers use that the network's input and output live on the
even sites), site counts below and beside the tiles of 8, 16 and 64 sites.  Loss and
every layer's gradient against the FP64 oracle: FP32 weights, activations and links and
sums of ~10^3 products, 1e-5 for the loss and 1e-4 (norm-relative, per layer) for the
gradient, as in test_gpu_ptc.py.
"""
import numpy as np
import pytest

from oracle import ptc
from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import relerr, setup
from tests.test_gpu_ptc import flat, rand_weights, unflat

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,cstar", [((2, 2, 2, 2), 0), ((2, 2, 4, 6), 1), ((2, 4, 6, 6), 0)])
@pytest.mark.parametrize("nlayers,nch", [(1, 4), (2, 1), (2, 8), (3, 2), (3, 5), (2, 16)])
def test_loss_and_gradient_by_layer(L, cstar, nlayers, nch):
    qxd, ctx, op, _, _ = setup(L, cstar, (np.pi, 0.0, 0.0, 0.0), qhat=4, seed=7400)
    Ws = rand_weights(np.random.default_rng(3), nlayers, nch)
    ne = op.geom.V // 2
    r = workload.spinor(ne, 7401, nrhs=2).astype(np.complex64)
    e = workload.spinor(ne, 7402, nrhs=2).astype(np.complex64)
    W32 = flat(Ws)
    grad = np.zeros_like(W32)
    loss = ctx.ptc_loss_grad(0, W32, nlayers, nch, r, e, 2, grad=grad, kind=qxd.LOSS_RESIDUAL)
    Wr = unflat(W32.astype(np.complex128), nlayers, nch)
    pairs = [(r[i].astype(np.complex128), e[i].astype(np.complex128)) for i in range(2)]
    L0, G = ptc.loss_and_grad(ptc.Transport(op), Wr, pairs, norm="residual")
    assert abs(loss - L0) <= 1e-5 * L0
    for got, ref in zip(unflat(grad.astype(np.complex128), nlayers, nch), G):
        assert relerr(got, ref) <= 1e-4
    ctx.close()
