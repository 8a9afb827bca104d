"""Solves whose kernels' blocks are placed while the kernel before drains: the
same results, bit for bit, as with ordinary launches (a profiled solve's), for
solves back to back in one workspace and replayed from a graph.
"""
import pytest
import torch

from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,shape,phi", [("mixed", (32, 36, 5), False), ("mixed", (64, 64, 64), True),
                                                 ("mixed", (405, 128, 40), False), ("mixed", (256, 256, 33), False),
                                                 ("mixed", (45, 2187, 3), False), ("refined", (64, 48, 5), True)])
def test_same_bits(precision, shape, phi):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 100.0))
    dev = torch.device("cuda", 0)
    dt = torch.float32 if precision == "mixed" else torch.float64
    gen = torch.Generator(device=dev)
    gen.manual_seed(3)
    ins = [tuple(torch.randn((nz + (c == 2), ny, nx), dtype=dt, device=dev, generator=gen) for c in range(3))
           for _ in range(6)]
    P = mp.Projector.from_grid(g, precision, dev)
    outs = [P.solve(*f, phi=phi) for f in ins]                    # back to back
    torch.cuda.synchronize()
    mp.monc_proj_profile(P.plan, True)
    want = [[t.clone() for t in P.solve(*f, phi=phi)] for f in ins]
    torch.cuda.synchronize()
    mp.monc_proj_profile(P.plan, False)
    for o, r in zip(outs, want):
        for a, b in zip(o, r):
            assert torch.equal(a, b)
    fields = tuple(t.clone() for t in ins[0])
    out = tuple(torch.empty_like(t) for t in fields)
    graph = torch.cuda.CUDAGraph()
    P.solve(*fields, out=out)
    torch.cuda.synchronize()
    with torch.cuda.graph(graph):
        P.solve(*fields, out=out)
    for f, r in zip(ins, want):
        for d, s in zip(fields, f):
            d.copy_(s)
        graph.replay()
        for a, b in zip(out, r):
            assert torch.equal(a, b)
    P.close()
