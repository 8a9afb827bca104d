"""FP32 BiCGStab on a column taller than a launch of eight-level tiles can be (65535 of
them): one iteration without a preconditioner against FP64 vectors, whose kernels
tests/test_gpu_krylov.py pins to the oracle; tolerances of tests/test_gpu_krylov_fp32.py.
"""
import pytest

from paper_2009_12849_gb300 import workloads as W
from tests.test_gpu_krylov import _mp, fp32_inputs, relmax, run

pytestmark = pytest.mark.gpu


def test_tall():
    mp = _mp()
    nz = 8 * 65535 + 9
    g = W.make_grid(4, 1, nz, 40.0, 30.0, W.uniform_dz(nz, 0.1))
    u, v, w = fp32_inputs(g, 5)
    ref, _, _, rr64 = run(g, u, v, w, 0.0, 1, "none")
    got, st, it, rr = run(g, u, v, w, 0.0, 1, "none", precision="mixed")
    assert st == mp.MONC_PROJ_ENOCONV and it == 1
    assert abs(rr - rr64) <= 2e-6 * rr64
    for a, b in zip(got, ref):
        assert relmax(a, b) < 4e-6
