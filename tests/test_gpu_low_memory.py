"""What a context does with less when the device has no memory left: clover leaves by slabs of one
slice, multi-shift corrections in groups, sweeps without the blocks' copies.  Results do not
depend on it.

16^4: the leaves of a slice take 7.3 MB (a slab holds one slice more than it serves), a half field
3.1 MB in FP32, the SAP copies 47 MB, a deflation vector 6.3 MB.
"""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)
L = (16, 16, 16, 16)
MB = 1 << 20


class Held:
    """All device memory but `left` bytes, held outside the context."""

    def __init__(self):
        self.parts = []

    def all_but(self, left):
        import torch
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        n = torch.cuda.mem_get_info()[0] - left
        assert n > 0
        self.parts.append(torch.empty(n, dtype=torch.uint8, device="cuda"))

    def __enter__(self):
        return self

    def __exit__(self, *exc):
        import torch
        self.parts.clear()
        torch.cuda.empty_cache()


def context(Ns):
    """Two flavours and the seeds of a subspace for the second, whose set-up has run once."""
    import torch
    qxd, ctx, op, _, _ = setup(L, 0, PI, kappa=0.126, device="cuda")
    ctx.set_clover(1, 4, 0.12, 1.9, 1.0)
    seeds = torch.randn(Ns, op.geom.V, 4, 3, dtype=torch.complex64, device="cuda")
    ctx.dfl_setup(1, seeds, Ns, ninv=0)
    ctx.set_clover(1, 4, 0.12, 1.9, 1.0)
    return qxd, ctx, op, seeds


@pytest.mark.parametrize("left", [18, 40])  # slabs of one slice; of four
def test_clover_leaves_by_small_slabs(left):
    import torch
    Ns = 16
    qxd, ctx, op, seeds = context(Ns)
    x = torch.from_numpy(workload.spinor(op.geom.V, 5)).cuda()
    want, out = torch.empty_like(x), torch.empty_like(x)
    ctx.apply_Dw(0, qxd.FP64, x, want)
    with Held() as held:
        held.all_but(60 * MB)
        ctx.dfl_setup(1, seeds, Ns, ninv=0)  # in the place of the leaves
        held.all_but(left * MB)
        ctx.set_clover(0, -2, 0.126, 1.90952, 1.0)
        ctx.apply_Dw(0, qxd.FP64, x, out)
        torch.cuda.synchronize()
    assert torch.equal(out, want)
    ctx.close()


@pytest.mark.parametrize("left", [30, 54])  # one shift at a time; two (of five)
def test_corrections_in_groups(left):
    import torch
    Ns = 32
    qxd, ctx, op, seeds = context(Ns)
    phi = torch.from_numpy(workload.spinor(op.geom.V // 2, 6)).cuda()
    sigma = np.geomspace(1e-2, 8.0, 5)
    want = torch.empty((5,) + tuple(phi.shape), dtype=phi.dtype, device="cuda")
    out = torch.empty_like(want)
    ctx.solve_multishift(0, sigma, phi, want, tol=1e-10, inner=qxd.FP32)
    with Held() as held:
        held.all_but(80 * MB)
        ctx.dfl_setup(1, seeds, Ns, ninv=0)  # in the place of the leaves and the corrections
        held.all_but(left * MB)
        info = ctx.solve_multishift(0, sigma, phi, out, tol=1e-10, inner=qxd.FP32)
    assert info.true_relres <= 1e-10
    assert torch.equal(out, want)
    ctx.close()


def test_sweeps_after_their_copies_are_given_back():
    import torch
    Ns = 24
    qxd, ctx, op, seeds = context(Ns)
    ctx.set_sap(2, 2)
    eta = torch.randn(op.geom.V, 4, 3, dtype=torch.complex64, device="cuda")
    want, out = torch.empty_like(eta), torch.empty_like(eta)
    ctx.sap_apply(0, eta, want)
    with Held() as held:
        held.all_but(20 * MB)
        ctx.dfl_setup(1, seeds, Ns, ninv=0)  # 151 MB: the leaves' 116 MB are not enough
        ctx.sap_apply(0, eta, out)
    assert torch.equal(out, want)
    ctx.close()
