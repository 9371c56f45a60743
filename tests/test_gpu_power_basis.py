"""Unpreconditioned FP32 inner solves from the shifted power basis.

Restart lengths on both sides of where the inner products split (8) and of where the
power basis ends (16), one step per cycle, a budget that ends within a cycle, an
operator proportional to the identity up to the site-diagonal term (a basis that is used
up after a few steps), and a residual almost in the operator's kernel.  Solutions are held
to the requested true residual with the FP64 oracle; the iteration count of a restart
length is that of GCR, whose iterates the method reproduces in exact arithmetic, to within
one cycle per outer step.
"""
import numpy as np
import pytest

from oracle import DiracOperator, Flavour, GaugeField, Geometry
from oracle.solvers import gcr
from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import need_gpu, setup

pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)


@pytest.mark.parametrize("nkv", [1, 2, 8, 9, 16, 17])
def test_restart_lengths(nkv):
    qxd, ctx, op, _, _ = setup((4, 4, 6, 8), 2, PI, qhat=4, kappa=0.12)
    eta = workload.spinor(op.geom.V, 5)
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-10 * np.linalg.norm(eta)
    if nkv >= 8:
        # the same even-odd system to the inner solve's 1e-5, then again to what is left
        ev, od = op.even_sites(), op.odd_sites()
        Dinv = op.Doo_inv()
        b = eta[ev] - op.Deo(np.einsum("nab,nb->na", Dinv, eta[od].reshape(-1, 12)).reshape(-1, 4, 3))
        _, its = gcr(lambda v: op.Dhat(v, Dinv), b, 1e-10, nkv, 1000)
        assert info.iters <= its + 2 * nkv
    short = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10, nmx=5, check=False)
    assert short.status == 2 and short.iters <= 5
    ctx.close()


@pytest.mark.parametrize("nkv", [8, 16])
def test_basis_that_is_used_up(nkv):
    # kappa -> 0: Dhat = 1/(2 kappa) up to a relative 1e-5, so one or two steps exhaust the basis
    qxd, ctx, op, _, _ = setup((4, 4, 4, 4), 0, PI, kappa=1e-5)
    eta = workload.spinor(op.geom.V, 6)
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    assert info.iters <= 4 * nkv
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-10 * np.linalg.norm(eta)
    zero = np.zeros_like(eta)
    ctx.solve(0, zero, psi, nkv=nkv, inner=qxd.FP32, tol=1e-10)
    assert not psi.any()
    ctx.close()


@pytest.mark.parametrize("nkv", [1, 2])
def test_residual_almost_in_the_kernel(nkv):
    # Free field, bare mass m0 = 5e-4.  On the even sites Dhat multiplies a constant spinor by
    # about 2 m0 and the mode (-1)^(x2 + x3), which the hopping term annihilates, by 1/(2 kappa).
    # The first cycle takes the second mode away and centres the powers on it; for what is
    # left |Dhat r|^2 is below the rounding of |d r|^2.
    kappa = 0.5 / (4 + 5e-4)
    L, zero = (8, 8, 8, 8), (0.0, 0.0, 0.0, 0.0)
    qxd = need_gpu()
    geom = Geometry(L, 0, zero)
    U = np.broadcast_to(np.eye(3, dtype=complex), (geom.V, 4, 3, 3)).copy()
    A = np.zeros((geom.V, 4))
    op = DiracOperator(GaugeField(geom, U, A, 6.0), Flavour(4, kappa, 1.0, 1.0))
    ctx = qxd.Context(L, 0, zero)
    ctx.set_links(U, A, 6.0)
    ctx.set_clover(0, 4, kappa, 1.0, 1.0)
    x = np.stack(np.unravel_index(np.arange(geom.V), L))
    lo = np.random.default_rng(3).standard_normal((4, 3))
    eta = (1 - x.sum(0) % 2)[:, None, None] * (((-1.0) ** (x[2] + x[3]))[:, None, None] + 0.1 * lo) + 0j
    psi = np.empty_like(eta)
    info = ctx.solve(0, eta, psi, nkv=nkv, inner=qxd.FP32, tol=1e-5)
    assert np.linalg.norm(eta - op.apply(psi)) <= 1e-5 * np.linalg.norm(eta)
    assert info.iters <= 20
    ctx.close()
