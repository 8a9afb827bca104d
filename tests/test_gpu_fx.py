"""FP64 plans' fixed-point transforms: lengths of every radix mix against the FP64
oracle (1e-12, the path's tolerance), inputs far from 1 in magnitude, of one
level or row only, zero, and with a NaN or an infinity.

A transform's elements share one scale (its largest element), so its error is
relative to the whole transform, as a floating-point transform's is.
"""
import numpy as np
import pytest
import torch

import oracle as O
from paper_2009_12849_gb300 import workloads as W
from tests.test_gpu_parity import check_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(36, 45, 3), (50, 1000, 2), (1000, 48, 2), (54, 625, 2), (625, 60, 2), (729, 72, 2),
                                   (75, 729, 2), (81, 80, 3), (125, 90, 3), (108, 120, 3), (96, 100, 3), (192, 135, 3),
                                   (243, 250, 2), (512, 40, 2), (40, 512, 2), (972, 96, 2), (800, 72, 2),
                                   (384, 36, 3), (36, 320, 3), (64, 64, 129), (128, 65 - 1, 33)])
def test_lengths(shape):
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 40.0))
    check_case(g, 5, True, "fp64")


def _solve(g, u, v, w, phi=True):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    P = mp.Projector.from_grid(g, "fp64", torch.device("cuda", 0))
    out = P.solve(*(torch.tensor(a, device="cuda") for a in (u, v, w)), phi=phi)
    torch.cuda.synchronize()
    assert P.sync_status() == 0
    res = [o.cpu().numpy() for o in out]
    P.close()
    return res


@pytest.mark.parametrize("scale", [1e-200, 1e-30, 1e30, 1e200])
def test_magnitudes(scale):
    """The projection is linear: scaled inputs give scaled outputs (powers of ten
    round, so to the path's tolerance)."""
    g = W.make_grid(64, 48, 7, 25.0, 20.0, W.geometric_dz(7, 10.0, 40.0))
    u, v, w = W.random_fields(g, 3, True)
    a = _solve(g, u, v, w)
    b = _solve(g, u * scale, v * scale, w * scale)
    for x, y in zip(a, b):
        assert np.linalg.norm(y / scale - x) <= 1e-12 * np.linalg.norm(x)


def test_uneven_magnitudes():
    """One quiet level and one quiet row beside strong ones, and zero input."""
    g = W.make_grid(72, 64, 6, 25.0, 20.0, W.geometric_dz(6, 10.0, 40.0))
    u, v, w = W.random_fields(g, 4, True)
    u[2] *= 1e-9
    v[2] *= 1e-9
    u[:, 5] *= 1e-9
    ref = O.project(u, v, w, g.dx, g.dy, g.dz, g.rho_c, g.rho_f)
    out = _solve(g, u, v, w, phi=False)
    a = np.concatenate([x.ravel() for x in out])
    b = np.concatenate([x.ravel() for x in ref[:3]])
    assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
    z = _solve(g, 0 * u, 0 * v, 0 * w)
    assert all(np.all(x == 0) for x in z)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_not_finite(bad):
    """A cell that is not finite reaches every column of its level's spectrum, and
    through the vertical solve every level, as in floating point."""
    g = W.make_grid(64, 48, 5, 25.0, 20.0, W.uniform_dz(5, 20.0))
    u, v, w = W.random_fields(g, 3, False)
    u[2, 7, 9] = bad
    out = _solve(g, u, v, w)
    assert np.all(np.isnan(out[0])) and np.all(np.isnan(out[1])) and np.all(np.isnan(out[2][1:-1]))
    assert np.all(out[2][0] == 0) and np.all(out[2][-1] == 0)
