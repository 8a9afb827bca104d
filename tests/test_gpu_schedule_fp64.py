"""monc_proj_plan_schedule of FP64 plans: the elements per thread that the plan's
kernels hold (405 = 9 9 5, 1000 = 10 10 10, 96 = 12 8; 16 for powers of two and for a
length without a compile-time plan).
"""
import pytest
import torch

from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,want", [(256, 64, (16, 16)), (405, 1000, (9, 10)), (96, 1536, (12, 16))])
def test_elements(nx, ny, want):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    g = W.make_grid(nx, ny, 2, 25.0, 25.0, W.uniform_dz(2, 20.0))
    P = mp.Projector.from_grid(g, "fp64", torch.device("cuda", 0))
    got = mp.monc_proj_plan_schedule(P.plan)
    P.close()
    assert (got["row_elems"], got["col_elems"]) == want
