"""Solves of one plan on several streams at once, each a chain of kernels whose
blocks are placed before the kernel before them counts as finished: the bits
of solves one after the other.
"""
import pytest
import torch

from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shape", [("mixed", (64, 64, 64)), ("mixed", (405, 128, 40)), ("mixed", (32, 36, 300)),
                                             ("refined", (64, 48, 5))])
def test_streams(precision, shape):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 100.0))
    dev = torch.device("cuda", 0)
    dt = torch.float32 if precision == "mixed" else torch.float64
    gen = torch.Generator(device=dev)
    gen.manual_seed(4)
    P = mp.Projector.from_grid(g, precision, dev)
    ins = [tuple(torch.randn((nz + (c == 2), ny, nx), dtype=dt, device=dev, generator=gen) for c in range(3))
           for _ in range(4)]
    want = [[t.clone() for t in P.solve(*f)] for f in ins]
    streams = [torch.cuda.Stream() for _ in ins]
    spaces = [torch.empty_like(P.workspace) for _ in ins]
    outs = [tuple(torch.empty_like(t) for t in f) for f in ins]
    torch.cuda.synchronize()
    for _ in range(20):
        for f, o, ws, st in zip(ins, outs, spaces, streams):
            mp.monc_proj_solve(P.plan, *f, *o, None, ws, st)
    torch.cuda.synchronize()
    assert P.sync_status() == 0
    for o, r in zip(outs, want):
        for a, b in zip(o, r):
            assert torch.equal(a, b)
    P.close()
