"""The operator kernels on canonical fields against the kernels on converted fields.

A field that is not 32-byte aligned takes the conversion path, an aligned one the
kernels that read and write it in place.  Both evaluate the same expression in the same
order, so the results are equal bit for bit; but up to 4096 (FP64) or 8192 (FP32) sites times
right-hand sides four lanes share a site and add in another order: two results that are
each within 1e-13 or 2e-6 of the exact one (test_gpu_operator.py) agree to twice that.
"""
import numpy as np
import pytest

from tests.gpu_helpers import relerr, setup

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

PI = (np.pi, 0.0, 0.0, 0.0)
# site counts below, at and beyond the tiles of 64 and 128 sites, odd block remainders, C* shifts
GEOMS = [((2, 2, 2, 2), 0), ((4, 2, 4, 2), 1), ((4, 6, 2, 10), 2), ((6, 4, 6, 4), 3), ((4, 4, 4, 4), 0),
         ((8, 8, 10, 14), 3)]


def _field(n, dtype, offset, seed):
    """A complex field of n numbers whose first byte is `offset` bytes beyond a 32-byte boundary."""
    gen = torch.Generator().manual_seed(seed)
    size = 16 if dtype == torch.complex128 else 8
    v = torch.view_as_complex(torch.randn(n + 4, 2, generator=gen, dtype=torch.float64)).to(dtype)[:n]
    buf = torch.zeros(n + 8, dtype=dtype, device="cuda")
    start = (-buf.data_ptr() // size) % (32 // size) + offset // size
    f = buf[start:start + n]
    f.copy_(v)
    assert f.data_ptr() % 32 == offset
    return f


@pytest.mark.parametrize("L,cstar", GEOMS)
@pytest.mark.parametrize("prec", [0, 1, 2])
@pytest.mark.parametrize("nrhs", [1, 3, 5])
def test_canonical_and_converted_fields_agree(L, cstar, prec, nrhs):
    qxd, ctx, op, _, _ = setup(L, cstar, PI, qhat=4, kappa=0.13)
    dtype = torch.complex128 if prec == 0 else torch.complex64
    for n, call in ((12 * op.geom.V, ctx.apply_Dw), (6 * op.geom.V, ctx.apply_Dhat_eo)):
        for kw in ({},) if call == ctx.apply_Dw else ({"dagger": False}, {"dagger": True}):
            outs = []
            for offset in (0, 16):
                x, y = _field(n * nrhs, dtype, offset, 3), _field(n * nrhs, dtype, offset, 4)
                call(0, prec, x, y, nrhs=nrhs, **kw)
                outs.append(y.cpu().numpy())
            sites = op.geom.V // (1 if call == ctx.apply_Dw else 2)
            if prec != 2 and sites * nrhs <= (4096 if prec == 0 else 8192):
                assert relerr(outs[0].astype(np.complex128), outs[1].astype(np.complex128)) <= (2e-13 if prec == 0 else 4e-6)
            else:
                assert np.array_equal(outs[0], outs[1])
            if call == ctx.apply_Dhat_eo:  # in place
                x = _field(n * nrhs, dtype, 0, 3)
                call(0, prec, x, x, nrhs=nrhs, **kw)
                assert np.array_equal(x.cpu().numpy(), outs[0])
    ctx.close()


def test_partly_overlapping_fields_take_the_converted_path():
    qxd, ctx, op, _, _ = setup((4, 4, 4, 4), 0, PI)
    n = 6 * op.geom.V
    ref = torch.empty(n, dtype=torch.complex64, device="cuda")
    x = _field(n, torch.complex64, 0, 3)
    ctx.apply_Dhat_eo(0, qxd.BF16, x, ref)
    buf = torch.empty(n + 4, dtype=torch.complex64, device="cuda")
    buf[:n].copy_(x)
    ctx.apply_Dhat_eo(0, qxd.BF16, buf[:n], buf[4:])
    assert torch.equal(buf[4:], ref)
    ctx.close()


@pytest.mark.parametrize("prec", [0, 1])
def test_small_lattice_calls_in_a_graph(prec):
    # launches that let the next one start early, recorded and replayed on new inputs
    qxd, ctx, op, _, _ = setup((4, 4, 4, 6), 1, PI, qhat=4, kappa=0.13)
    n = 6 * op.geom.V
    dtype = torch.complex128 if prec == 0 else torch.complex64
    x, y, z = _field(n, dtype, 0, 3), _field(n, dtype, 0, 4), _field(n, dtype, 0, 5)
    ctx.apply_Dhat_eo(0, prec, x, y)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        st = torch.cuda.current_stream()
        for _ in range(3):
            ctx.apply_Dhat_eo(0, prec, x, y, stream=st)
            ctx.apply_Dhat_eo(0, prec, y, z, dagger=True, stream=st)
    x.copy_(_field(n, dtype, 0, 6))
    graph.replay()
    torch.cuda.synchronize()
    got = [y.clone(), z.clone()]
    ctx.apply_Dhat_eo(0, prec, x, y)
    ctx.apply_Dhat_eo(0, prec, y, z, dagger=True)
    assert torch.equal(got[0], y) and torch.equal(got[1], z)
    ctx.close()
