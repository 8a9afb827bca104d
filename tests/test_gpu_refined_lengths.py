"""Refined plans at horizontal lengths that have compile-time FP32 kernels but
not all of the refinement passes' own: every kernel of the plan must follow
one radix plan.  FP64 oracle, the refined path's 1e-12.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(200, 200, 6), (64, 135, 5), (135, 64, 5), (64, 48, 5), (500, 300, 3), (40, 640, 2)])
def test_refined(shape):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 100.0))
    u, v, w = W.random_fields(g, 5, True)
    ref = O.project(u, v, w, g.dx, g.dy, g.dz, g.rho_c, g.rho_f)
    P = mp.Projector.from_grid(g, "refined", torch.device("cuda", 0))
    out = P.solve(*(torch.tensor(a, device="cuda") for a in (u, v, w)))
    torch.cuda.synchronize()
    assert P.sync_status() == 0
    a = np.concatenate([x.cpu().numpy().ravel() for x in out])
    b = np.concatenate([x.ravel() for x in ref[:3]])
    assert np.linalg.norm(a - b) < 1e-12 * np.linalg.norm(b)
    P.close()
