"""FP64 plans on smooth fields: one large-scale mode, whose spectrum is a few
large coefficients.  White noise (the other tests' fields) grows through a
transform's stages and hides bits that a fixed-point stage takes off;
a single mode does not.

What is left of the potential, and of a field that is a pure gradient, after
the mode itself (least squares, so that the last bits of the wavenumbers'
tables do not count) is the transforms' error.  Tolerance 3e-16 of the mode:
two transforms (columns, rows) of 1.5e-16 at most for any data (fx.cuh), three
roundings to doubles (input, columns' and rows' results, 0.45e-16 rms each).
FP64 butterflies reach 1e-16 each.
"""
import math

import numpy as np
import pytest
import torch

from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def rest(x, c, s):
    """rms of x without its part in the span of c and s."""
    n = x.size
    m = np.array([[np.sum(c * c), np.sum(c * s)], [np.sum(c * s), np.sum(s * s)]])
    a = np.linalg.solve(m, [np.sum(x * c), np.sum(x * s)])
    return math.sqrt(float(np.sum((x - a[0] * c - a[1] * s) ** 2)) / n)


@pytest.mark.parametrize("nx,ny", [(360, 405), (405, 360), (1000, 1024), (1024, 1000), (972, 256), (64, 625)])
@pytest.mark.parametrize("mx,my", [(1, 1), (3, 0), (0, 2)])
def test_one_mode(nx, ny, mx, my):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    g = W.make_grid(nx, ny, 1, 25.0, 20.0, W.uniform_dz(1, 20.0))
    # the angle in whole parts of a turn, so that it is exact before cos and sin
    part = (mx * ny * np.arange(nx)[None, :] + my * nx * np.arange(ny)[:, None]) % (nx * ny)
    th = 2 * np.pi * part.astype(np.longdouble) / (nx * ny)
    c, s = np.cos(th), np.sin(th)
    p = 3.0 * c + 1.0 * s
    u = (np.roll(p, -1, axis=1) - p) / g.dx
    v = (np.roll(p, -1, axis=0) - p) / g.dy
    c, s, u, v = (a.astype(np.float64) for a in (c, s, u, v))
    dev = torch.device("cuda", 0)
    P = mp.Projector.from_grid(g, "fp64", dev)
    tu, tv = (torch.tensor(a[None].copy(), device=dev) for a in (u, v))
    uo, vo, _, phi = (t.cpu().numpy() for t in
                      P.solve(tu, tv, torch.zeros((2, ny, nx), dtype=torch.float64, device=dev), phi=True))
    P.close()
    assert rest(phi[0], c, s) <= 3e-16 * math.sqrt(5.0)      # rms of p: sqrt((9 + 1) / 2)
    rms = math.sqrt(float(np.mean(u ** 2) + np.mean(v ** 2)))
    for got in (uo, vo):
        assert rest(got[0], c, s) <= 3e-16 * rms


@pytest.mark.parametrize("nx,ny", [(135, 200), (200, 135), (360, 90), (96, 100), (256, 64)])
def test_mean_flux(nx, ny):
    """The horizontal mean of the projected w is zero on every face: a bias in the
    transforms' roundings adds up there.  Noise of rms 1: the weighted divergence
    has rms 1.6, its spectrum's mean an error of 2.1e-16 (two transforms of 1.5e-16) of
    that per level, added up over half the 64 levels from either end: 1.5e-16 * 1.6 *
    1.4 * 8 / sqrt(nx ny) of the mean at most; four times that."""
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    nz = 64
    g = W.make_grid(nx, ny, nz, 25.0, 25.0, W.uniform_dz(nz, 10.0))
    u, v, w = (torch.tensor(a, device="cuda") for a in W.random_fields(g, nx))
    P = mp.Projector.from_grid(g, "fp64", torch.device("cuda", 0))
    wo = P.solve(u, v, w)[2].cpu().numpy()
    P.close()
    mean = wo.astype(np.longdouble).mean(axis=(1, 2))
    assert float(np.max(np.abs(mean))) <= 4 * 2.1e-16 * 1.6 * 8 / math.sqrt(nx * ny)
