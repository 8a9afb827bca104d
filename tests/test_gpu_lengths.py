"""Mixed solves at compile-time lengths past 512 and below 64 (shortest, longest,
odd, prime powers, many stages), against the FP64 oracle at the mixed path's
tolerances (1e-5 relative, divergence residual 1e-6; FP32 rounding of inputs shared).
"""
import pytest

from paper_2009_12849_gb300 import workloads as W
from tests.test_gpu_parity import check_case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(36, 2048, 2), (2048, 36, 2), (729, 125, 2), (125, 729, 2), (1875, 45, 2),
                                   (45, 1875, 2), (625, 81, 3), (81, 1458, 2), (2025, 50, 2), (768, 640, 2),
                                   (972, 75, 2), (54, 1080, 3)])
def test_lengths(shape):
    nx, ny, nz = shape
    g = W.make_grid(nx, ny, nz, 25.0, 20.0, W.geometric_dz(nz, 10.0, 40.0))
    check_case(g, 5, True, "mixed")
