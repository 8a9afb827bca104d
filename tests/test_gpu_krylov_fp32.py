"""BiCGStab on FP32 vectors where its kernels change: stencil four columns wide or
one (nx a multiple of 4 or not, more than one block along x, a part of one),
update four points wide or one, line sweeps with the column in shared memory
(one batch of levels, several, more than the default 48 KB) and in separate
kernels (a column that does not fit, and one that leaves few blocks on an SM where there
are many).  FP64 oracle after a fixed number of iterations on the same inputs.

Tolerance 4e-6 of the largest value, 2e-6 on the residual: FP32 vectors with
FP64 sums differ from FP64 by at most 3e-7 and 1e-7 on these grids (the same
method in numpy); the kernels' order of additions differs.
"""
import numpy as np
import pytest

import oracle.krylov as K
from paper_2009_12849_gb300 import workloads as W
from tests.test_gpu_krylov import _mp, fp32_inputs, grid, relmax, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precond", ["line", "none"])
@pytest.mark.parametrize("shape", [(27, 15, 33), (144, 6, 50), (300, 5, 17), (6, 5, 129), (12, 6, 200), (9, 8, 300),
                                   (8, 4, 830), (180, 160, 254)])
def test_fp32_grids(shape, precond):
    mp = _mp()
    g = grid(*shape)
    u, v, w = fp32_inputs(g, 27)
    iters = 3 if g.nx * g.ny * g.nz < 10 ** 6 else 1
    ref = K.project_krylov(u, v, w, g.dx, g.dy, g.dz, g.rho_c, g.rho_f, 0.0, iters, precond)
    got, st, it, rr = run(g, u, v, w, 0.0, iters, precond, precision="mixed")
    assert st == mp.MONC_PROJ_ENOCONV and it == iters
    assert abs(rr - ref[5]) <= 2e-6 * ref[5]
    for a, b in zip(got, ref[:4]):
        assert relmax(a, b) < 4e-6
    assert np.all(got[2][0] == 0) and np.all(got[2][-1] == 0)
