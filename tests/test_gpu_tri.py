"""The FP32 vertical solve alone (monc_proj_vertical_pencil) against a FP64 Thomas
solve of every column, at the level counts and spectral widths where its
split into warps and column groups changes: one warp, full and partial warps,
16 and 32 levels per warp, the sweeps past 256 levels, rows whose last columns
are gathered from several rows, rows that do not fill a group, both kinds of
columns in one group.

Tolerance 1e-5 (relative, the mixed path's): the columns' elimination is
backward stable in FP32 with a condition of at most 51 (|lambda| >= 0.02 v_max),
so a few units of 51 * 6e-8; the near-zero ones run on pairs.
"""
import numpy as np
import pytest
import torch

from paper_2009_12849_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def columns64(g, d):
    """p and its vertical face gradient of rho_c dz-weighted right-hand sides d (FP64)."""
    nx, ny, nz = g.nx, g.ny, g.nz
    zf = np.concatenate([[0.0], np.cumsum(g.dz)])
    dzn = np.diff(0.5 * (zf[1:] + zf[:-1]))
    a = np.zeros(nz + 1)
    a[1:nz] = g.rho_f[1:nz] / dzn
    s = g.rho_c * g.dz
    kx, ky = np.arange(nx // 2 + 1), np.arange(ny)
    lam = -4 * np.sin(np.pi * kx / nx)[None, :] ** 2 / g.dx ** 2 - 4 * np.sin(np.pi * ky / ny)[:, None] ** 2 / g.dy ** 2
    y, e = np.empty_like(d), np.empty(d.shape)
    for k in range(nz):
        e[k] = lam * s[k] - a[k] - a[k + 1]
        y[k] = d[k]
        if k:
            e[k] -= a[k] ** 2 * ie
            y[k] -= a[k] * ie * y[k - 1]
        with np.errstate(divide="ignore"):
            ie = 1.0 / e[k]
        if k == 0:
            ie[0, 0] = 0.0
        e[k] = ie
        if k == 0:
            y[0, 0, 0] = 0.0
    p = np.empty_like(d)
    p[-1] = y[-1] * e[-1]
    for k in range(nz - 2, -1, -1):
        p[k] = (y[k] - a[k + 1] * p[k + 1]) * e[k]
    gz = np.zeros_like(p)
    if nz > 1:
        gz[1:] = (p[1:] - p[:-1]) / dzn[:, None, None]
    return p / (nx * ny), gz / (nx * ny)


@pytest.mark.parametrize("nx,ny", [(64, 10), (96, 5), (40, 9), (30, 6), (16, 8), (6, 5), (1, 4)])
@pytest.mark.parametrize("nz", [1, 2, 7, 8, 16, 17, 32, 33, 100, 128, 129, 255, 256, 257])
def test_columns(nx, ny, nz):
    import __graft_entry__ as ge
    ge.build()
    from paper_2009_12849_gb300 import monc_proj as mp
    g = W.make_grid(nx, ny, nz, 20.0, 30.0, W.geometric_dz(nz, 10.0, 40.0))
    dev = torch.device("cuda", 0)
    P = mp.Projector.from_grid(g, "mixed", dev)
    nxp = mp.monc_proj_spectral_pitch(P.plan)
    rng = np.random.default_rng(nx * 1000 + nz)
    nxh = nx // 2 + 1
    d = (rng.standard_normal((nz, ny, nxh)) + 1j * rng.standard_normal((nz, ny, nxh))).astype(np.complex64)
    # the mean column's right-hand side sums to zero, as a divergence's does
    d[:, 0, 0] -= d[:, 0, 0].mean()
    spec = torch.zeros((nz, ny, nxp), dtype=torch.complex64, device=dev)
    spec[:, :, :nxh] = torch.from_numpy(d).to(dev)
    gz = torch.zeros_like(spec)
    mp.monc_proj_vertical_pencil(P.plan, 0, ny, spec, gz, P.workspace)
    torch.cuda.synchronize()
    assert P.sync_status() == 0
    p64, gz64 = columns64(g, d.astype(np.complex128))
    got = spec[:, :, :nxh].cpu().numpy()
    assert np.linalg.norm(got - p64) <= 1e-5 * np.linalg.norm(p64)
    if nz > 1:
        got = gz[1:, :, :nxh].cpu().numpy()
        assert np.linalg.norm(got - gz64[1:]) <= 1e-5 * np.linalg.norm(gz64[1:])
    P.close()
