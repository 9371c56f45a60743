"""Unpreconditioned FP32 inner solves at the ends of the power basis: sources far from 1 in
size, and operators and sources whose powers are no basis."""
import numpy as np
import pytest

from oracle import DiracOperator, Flavour, GaugeField, Geometry
from oracle.solvers import gcr
from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import need_gpu, setup

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


@pytest.mark.parametrize("L,m0,nkv", [((4, 4, 4, 4), 5e-4, 8), ((4, 4, 4, 4), 5e-4, 16), ((8, 4, 4, 4), 5e-3, 16)])
def test_powers_of_few_eigenvalues(L, m0, nkv):
    # Free field, bare mass m0: Dhat has a few distinct eigenvalues, about 2 m0 on constant spinors.
    # The powers of a source that is mostly constant are parallel to FP32 precision after a few
    # steps, while the steps of GCR go on reducing the residual.
    kappa = 0.5 / (4 + m0)
    zero = (0.0, 0.0, 0.0, 0.0)
    qxd = need_gpu()
    geom = Geometry(L, 0, zero)
    U = np.broadcast_to(np.eye(3, dtype=complex), (geom.V, 4, 3, 3)).copy()
    A = np.zeros((geom.V, 4))
    op = DiracOperator(GaugeField(geom, U, A, 6.0), Flavour(4, kappa, 1.0, 1.0))
    ctx = qxd.Context(L, 0, zero)
    ctx.set_links(U, A, 6.0)
    ctx.set_clover(0, 4, kappa, 1.0, 1.0)
    ev = op.even_sites()
    lo = np.random.default_rng(3).standard_normal((4, 3))
    b = lo + 0.1 * workload.spinor(geom.V // 2, 5)
    eta = np.zeros((geom.V, 4, 3), dtype=complex)
    eta[ev] = b
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-9)
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-9 * np.linalg.norm(eta)
    # an FP32 solve leaves about 1e-7 times the condition number, 4 / m0, of its source
    assert info.restarts <= 2
    if nkv == 16:
        # GCR to the inner solves' 1e-5 as often, and two cycles for FP32 rounding
        Dinv = op.Doo_inv()
        its = 0
        for _ in range(1 + info.restarts):
            x, n = gcr(lambda v: op.Dhat(v, Dinv), b, 1e-5, nkv, 1000)
            b = b - op.Dhat(x, Dinv)
            its += n
        assert info.iters <= its + 2 * nkv
    ctx.close()
