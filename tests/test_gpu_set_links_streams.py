"""New links while operators of the old ones are still queued on another stream.

The operators are asynchronous and streams of PyTorch do not wait for the default
stream, so qxd_set_links itself has to wait before it overwrites the links.
"""
import numpy as np
import pytest

from paper_1908_11673_gb300 import workload
from tests.gpu_helpers import setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,where", [(0, "other"), (1, "other"), (1, "same"), (1, "graph")])
def test_queued_operators_see_their_links(prec, where):
    import torch
    L = (16, 16, 16, 16)
    qxd, ctx, op, U, A = setup(L, 0, (np.pi, 0.0, 0.0, 0.0), kappa=0.13, device="cuda")
    U2, A2 = (torch.from_numpy(f).cuda() for f in workload.gauge_field(L, 2000, device="cuda"))
    dt = torch.complex128 if prec == 0 else torch.complex64
    x = torch.from_numpy(workload.spinor(op.geom.V, 5, nrhs=12)).to(dt).cuda()
    want, out = torch.empty_like(x), torch.empty_like(x)
    ctx.apply_Dw(0, prec, x, want, nrhs=12)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    links = None if where == "other" else s
    if where == "graph":  # recorded on s, run on another stream
        graph, run = torch.cuda.CUDAGraph(), torch.cuda.Stream()
        with torch.cuda.graph(graph, stream=s):
            ctx.apply_Dw(0, prec, x, out, nrhs=12, stream=s)
        with torch.cuda.stream(run):
            for _ in range(300):
                graph.replay()
    else:
        for _ in range(300):  # 20 ms and more of work; the last application counts
            ctx.apply_Dw(0, prec, x, out, nrhs=12, stream=s)
    ctx.set_links(U2, A2, stream=links)
    ctx.set_clover(0, -2, 0.12, 1.9, 1.0)
    torch.cuda.synchronize()
    assert torch.equal(out, want)
    ctx.apply_Dw(0, prec, x, out, nrhs=12)
    assert not torch.equal(out, want)
    ctx.close()
