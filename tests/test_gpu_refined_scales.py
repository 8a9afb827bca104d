"""Refined plans on fields far from 1 m/s: the divergence is rounded to FP32 by
integer arithmetic within the normal FP32 range and by the hardware's
conversion outside it.  FP64 oracle, the refined path's 1e-12 (the projection
is linear).
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 40, 5), (45, 64, 3)])
@pytest.mark.parametrize("exponent", [-40, -20, 0, 60, None])
def test_scaled_fields(shape, exponent):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    nx, ny, nz = shape
    scale = 0.0 if exponent is None else 2.0 ** exponent
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 100.0))
    u, v, w = W.random_fields(g, 7, True)
    ref = O.project(u, v, w, g.dx, g.dy, g.dz, g.rho_c, g.rho_f)
    P = mp.Projector.from_grid(g, "refined", torch.device("cuda", 0))
    out = P.solve(*(torch.tensor(a * scale, device="cuda") for a in (u, v, w)), phi=True)
    torch.cuda.synchronize()
    assert P.sync_status() == 0
    a = np.concatenate([x.cpu().numpy().ravel() for x in out[:3]])
    b = scale * np.concatenate([x.ravel() for x in ref[:3]])
    assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    P.close()
