"""The SAP sweep from the blocks' own copies of links and terms and from the fields.

Both read the same values (the phase is multiplied into the link by the same code) and
evaluate the same expressions, so the results are equal bit for bit; a new SW term
replaces the copies.
"""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("L,cstar", [((8, 8, 8, 8), 0), ((8, 8, 16, 8), 3)])
def test_sweeps_from_copies_and_from_fields(L, cstar, monkeypatch):
    qxd, ctx, op, _, _ = setup(L, cstar, (np.pi, 0.0, 0.0, 0.0), qhat=4, kappa=0.13)
    ctx.set_sap(2, 3)
    eta = workload.spinor(op.geom.V, 5).astype(np.complex64)
    out = [np.empty_like(eta) for _ in range(3)]
    ctx.sap_apply(0, eta, out[0])
    monkeypatch.setenv("QXD_SAP_BLOCKS", "0")
    ctx.sap_apply(0, eta, out[1])
    assert np.array_equal(out[0], out[1])
    ctx.set_clover(0, 4, 0.12, 1.9, 1.0)  # another operator in the same slot
    ctx.sap_apply(0, eta, out[1])
    monkeypatch.delenv("QXD_SAP_BLOCKS")
    ctx.sap_apply(0, eta, out[2])
    assert np.array_equal(out[1], out[2]) and not np.array_equal(out[0], out[2])
    ctx.close()
