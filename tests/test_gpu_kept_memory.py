"""Device memory that a context keeps between calls is there for its other calls."""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)


@pytest.mark.parametrize("shifts,Ns", [(0, 16), (10, 32)])
def test_workspaces_that_hold_nothing_are_given_back(shifts, Ns):
    # On 16^4 the clover leaves keep 116 MB and the corrections of ten shifts 189 MB; the deflation
    # basis takes 101 MB (Ns = 16) or 201 MB (32).  All but 64 MB of the device is held elsewhere.
    import torch
    qxd, ctx, op, _, _ = setup((16, 16, 16, 16), 0, PI, kappa=0.126, device="cuda")
    V = op.geom.V
    seeds = torch.randn(Ns, V, 4, 3, dtype=torch.complex64, device="cuda")
    ctx.dfl_setup(0, seeds, Ns, ninv=0)  # the workspaces of the set-up itself
    ctx.set_clover(0, -2, 0.126, 1.9, 1.0)  # drops the basis
    if shifts:
        phi = torch.randn(V // 2, 4, 3, dtype=torch.complex128, device="cuda")
        x = torch.empty(shifts, V // 2, 4, 3, dtype=torch.complex128, device="cuda")
        ctx.solve_multishift(0, np.geomspace(1e-2, 8.0, shifts), phi, x, tol=1e-9, inner=qxd.FP32)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    held = torch.empty(torch.cuda.mem_get_info()[0] - (64 << 20), dtype=torch.uint8, device="cuda")
    try:
        ctx.dfl_setup(0, seeds, Ns, ninv=0)
    finally:
        held = None
        torch.cuda.empty_cache()
    out = torch.empty(V, 4, 3, dtype=torch.complex64, device="cuda")
    ctx.dfl_basis(0, 0, out)
    assert abs(float(torch.linalg.vector_norm(out)) - np.sqrt(V / 256)) < 1e-3  # norm 1 on every block
    ctx.close()


def test_sap_copies_keep_their_buffer(monkeypatch):
    # a new term or a new gauge field fills the buffer again: nothing is freed and allocated for it
    import torch
    L = (16, 16, 16, 16)
    qxd, ctx, op, _, _ = setup(L, 0, PI, kappa=0.126, device="cuda")
    U, A = (torch.from_numpy(f).cuda() for f in workload.gauge_field(L, 2000, device="cuda"))
    ctx.set_sap(1, 2)
    eta = torch.randn(op.geom.V, 4, 3, dtype=torch.complex64, device="cuda")
    copies, fields = torch.empty_like(eta), torch.empty_like(eta)

    def used():
        torch.cuda.synchronize()
        free, total = torch.cuda.mem_get_info()
        return total - free

    def sweep():
        ctx.sap_apply(0, eta, copies)
        with monkeypatch.context() as m:
            m.setenv("QXD_SAP_BLOCKS", "0")
            ctx.sap_apply(0, eta, fields)
        assert torch.equal(copies, fields)

    sweep()
    held = used()
    ctx.set_clover(0, -2, 0.12, 1.9, 1.0)
    assert used() == held
    sweep()
    ctx.set_links(U, A)
    ctx.set_clover(0, -2, 0.12, 1.9, 1.0)
    assert used() == held
    sweep()
    assert used() == held
    ctx.close()
