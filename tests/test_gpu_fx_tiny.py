"""FP64 plans on fields below the normal range of doubles: results keep the bits
that such numbers have, as FP64 arithmetic's do.
"""
import numpy as np
import pytest

from paper_2009_12849_gb300 import workloads as W
from tests.test_gpu_fx import _solve

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 64, 7), (72, 48, 7)])
def test_below_the_normal_range(shape):
    """Fields of 2^-1030, whose values hold 44 bits in units of 2^-1074.  An element of the
    spectra is rounded to such a unit, so its transform by up to 64 units (the root of the
    cells of a level): 64 * 2^-44 of the correction."""
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 40.0))
    u, v, w = W.random_fields(g, 3, True)
    t = 2.0 ** -1030
    u, v, w = (a * t / t for a in (u, v, w))             # as they are after rounding
    a = _solve(g, u, v, w)
    b = _solve(g, u * t, v * t, w * t)
    for x, y, f in zip(a, b, (u, v, w, 0.0)):
        assert np.linalg.norm(y / t - x) <= 64 * 2.0 ** -44 * np.linalg.norm(x - f)
