"""Representative calls of the projection library: what a model that uses it runs.

Each case is one call of a public entry point on a grid of the sizes that the
library's workloads, its server and its batch recipe use, or of the ragged
2^a 3^b 5^c sizes that a model's own domain brings.  ``prepare`` makes what a
model holds between steps (fields on the device, a plan with its workspace,
output arrays), ``run`` is one call, ``exact`` is the same result in 64 bits by
plain torch.
"""
from __future__ import annotations

import math

import torch

from paper_2009_12849_gb300 import monc_proj as MP
from paper_2009_12849_gb300 import workloads as W

KRYLOV_ITERS = 8


def _solve(name, precision, nx, ny, nz, dx, dz0, dz1, phi=False):
    return {"name": name, "kind": "solve", "precision": precision, "nx": nx, "ny": ny, "nz": nz,
            "dx": dx, "dy": dx, "dz0": dz0, "dz1": dz1, "phi": phi}


def listed():
    return [
        # the smallest workload: a 64-cube of a convective boundary layer, once per
        # time step of a small model, where launches and latency count
        _solve("mixed_64x64x64", "mixed", 64, 64, 64, 50.0, 25.0, 25.0),
        # the same in double precision, as the workload is specified
        _solve("fp64_64x64x64", "fp64", 64, 64, 64, 50.0, 25.0, 25.0),
        # an ordinary domain, with the potential kept as a diagnostic
        _solve("mixed_256x256x128_phi", "mixed", 256, 256, 128, 25.0, 10.0, 100.0, phi=True),
        # the same domain in double precision
        _solve("fp64_256x256x128", "fp64", 256, 256, 128, 25.0, 10.0, 100.0),
        # the headline workload and the largest call
        _solve("mixed_1024x1024x256", "mixed", 1024, 1024, 256, 10.0, 5.0, 50.0),
        # a served request: odd horizontal size, odd number of levels
        _solve("mixed_405x405x93", "mixed", 405, 405, 93, 25.0, 10.0, 100.0),
        # an uneven domain, longer than the sizes the server draws
        _solve("mixed_768x640x72", "mixed", 768, 640, 72, 20.0, 10.0, 80.0),
        # a ragged double-precision domain
        _solve("fp64_360x300x75", "fp64", 360, 300, 75, 25.0, 10.0, 100.0),
        # double-precision fields by the refined solver (three mixed passes)
        _solve("refined_512x512x96", "refined", 512, 512, 96, 20.0, 10.0, 60.0),
        # the second pressure solver in single precision with a fixed budget of
        # iterations
        {"name": "krylov_256x256x128", "kind": "krylov", "precision": "mixed", "nx": 256, "ny": 256, "nz": 128,
         "dx": 25.0, "dy": 25.0, "dz0": 10.0, "dz1": 100.0, "phi": True},
        # an uneven batch of independent domains (an ensemble) in one call
        {"name": "batch_16", "kind": "batch", "precision": "mixed", "count": 16, "recipe": 3, "grouped": True},
        # a model that keeps its fields on the host: page-locked arrays in and out
        {"name": "host_256x256x128", "kind": "host", "precision": "mixed", "nx": 256, "ny": 256, "nz": 128,
         "dx": 25.0, "dy": 25.0, "dz0": 10.0, "dz1": 100.0, "phi": False},
    ]


# points of the largest drawn grid, so that none costs more than the headline workload
_MOST = {"mixed": 48 << 20, "fp64": 6 << 20, "refined": 16 << 20, "krylov": 8 << 20, "host": 16 << 20}


def draw(rng):
    what = rng.choice(["mixed"] * 5 + ["fp64"] * 3 + ["refined", "krylov", "batch", "host"])
    if what == "batch":
        return {"kind": "batch", "precision": "mixed", "count": rng.randint(4, 16), "recipe": rng.randint(10, 10 ** 6),
                "grouped": rng.random() < 0.7}
    most = _MOST[what]
    sizes = [n for n in W.smooth_sizes(2048) if n >= 32]
    near = lambda x: min(sizes, key=lambda n: (abs(n - x), n))  # noqa: E731
    while True:
        nx = near(math.exp(rng.uniform(math.log(32), math.log(1536))))
        ny = nx if rng.random() < 0.5 else near(nx * math.exp(rng.uniform(-0.7, 0.7)))
        nz = int(round(math.exp(rng.uniform(math.log(24), math.log(256)))))
        if nx * ny * nz <= most:
            break
    dx = rng.choice([10.0, 25.0, 50.0])
    dz0 = rng.choice([5.0, 10.0, 25.0])
    return {"kind": what if what in ("krylov", "host") else "solve",
            "precision": what if what in ("fp64", "refined") else "mixed", "nx": nx, "ny": ny, "nz": nz,
            "dx": dx, "dy": dx, "dz0": dz0, "dz1": dz0 * rng.choice([1.0, 4.0, 10.0]),
            "phi": what in ("mixed", "fp64", "refined", "krylov") and rng.random() < 0.3}


def _grid(case):
    return W.make_grid(case["nx"], case["ny"], case["nz"], case["dx"], case["dy"],
                       W.geometric_dz(case["nz"], case["dz0"], case["dz1"]))


def _grids(case):
    if case["kind"] == "batch":
        return [g for g, _ in W.batch_instances(case["count"], case["recipe"])]
    return [_grid(case)]


def _fields(g, dtype, gen):
    """Turbulent provisional velocities: N(0,1) in every cell on a 1 m/s mode of the
    domain's size; w vanishes at the bottom and top faces."""
    dev = torch.device("cuda")

    def axis(n, off):
        return (torch.arange(n, device=dev, dtype=torch.float64) + off) / n

    zf = torch.from_numpy(W.face_heights(g.dz)).to(dev)
    zc = 0.5 * (zf[:-1] + zf[1:])

    def field(xo, yo, z):
        f = torch.randn((len(z), g.ny, g.nx), dtype=dtype, device=dev, generator=gen)
        hor = torch.cos(2 * math.pi * axis(g.ny, yo))[:, None] * torch.sin(2 * math.pi * axis(g.nx, xo))[None, :]
        return f.addcmul_(torch.sin(math.pi * z / zf[-1]).to(dtype)[:, None, None], hor.to(dtype)[None])

    u, v, w = field(1.0, 0.5, zc), field(0.5, 1.0, zc), field(0.5, 0.5, zf)
    w[0].zero_()
    w[-1].zero_()
    return u, v, w


def _inputs(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    dtype = MP.DTYPES[MP.PRECISIONS[case["precision"]]]
    grids = _grids(case)
    return grids, [_fields(g, dtype, gen) for g in grids]


def _host_like(t):
    return torch.empty(t.shape, dtype=t.dtype, pin_memory=True)


def prepare(case, seed):
    grids, fields = _inputs(case, seed)
    outs = [tuple(torch.empty_like(t) for t in f) for f in fields]
    s = {"case": case, "in": fields, "out": outs}
    if case["kind"] == "batch":
        s["proj"] = MP.BatchProjector(grids, case["precision"])
        s["fields"] = [f + o for f, o in zip(fields, outs)]
        return s
    s["proj"] = MP.Projector.from_grid(grids[0], case["precision"])
    if case["kind"] == "krylov":
        s["workspace"] = torch.empty(MP.monc_proj_krylov_workspace_size(s["proj"].plan), dtype=torch.uint8,
                                     device="cuda")
    elif case["kind"] == "host":
        s["in"] = [tuple(_host_like(t).copy_(t) for t in fields[0])]
        s["out"] = [tuple(_host_like(t) for t in fields[0])]
        s["staging"] = torch.empty(MP.monc_proj_host_staging_size(s["proj"].plan), dtype=torch.uint8, device="cuda")
    return s


def run(state):
    case, proj = state["case"], state["proj"]
    if case["kind"] == "batch":
        proj.solve(state["fields"], grouped=case["grouped"])
        return [list(o) for o in state["out"]]
    (u, v, w), out = state["in"][0], state["out"][0]
    if case["kind"] == "host":
        return list(proj.solve_host(u, v, w, out, staging=state["staging"]))
    if case["kind"] == "krylov":
        uo, vo, wo, phi, _, iters, _ = proj.solve_krylov(u, v, w, tol=0.0, max_iter=KRYLOV_ITERS, precond="line",
                                                         out=out, phi=case["phi"], workspace=state["workspace"])
        return {"u": uo, "v": vo, "w": wo, "phi": phi, "iterations": iters}
    return list(proj.solve(u, v, w, out=out, phi=case["phi"]))


def work(case):
    elem = 8 if case["precision"] in ("fp64", "refined") else 4
    nbytes = flops = 0
    for g in _grids(case):
        n = g.nx * g.ny * g.nz
        face = g.nx * g.ny
        nbytes += elem * (6 * n + 2 * face + (n if case.get("phi") else 0))
        if case["kind"] == "krylov":
            # two stencils, two line solves and the vector updates of an iteration
            flops += n * (13 + 60 * KRYLOV_ITERS)
        else:
            # one forward and three inverse real transforms each way, the vertical solve,
            # the divergence and the correction
            flops += n * (10 * math.log2(max(2, g.nx * g.ny)) + 24)
    return {"bytes": nbytes, "flops": flops}


# ---------------------------------------------------------------- 64-bit values


class _Op:
    """Discrete operators of one grid in 64 bits."""

    def __init__(self, g):
        dev = torch.device("cuda")
        t = lambda a: torch.tensor(a, dtype=torch.float64, device=dev)  # noqa: E731
        self.nx, self.ny, self.nz, self.dx, self.dy = g.nx, g.ny, g.nz, g.dx, g.dy
        self.dz, self.rc, self.rf = t(g.dz), t(g.rho_c), t(g.rho_f)
        self.dzn = 0.5 * (self.dz[1:] + self.dz[:-1])               # interior faces
        self.a = torch.zeros(g.nz + 1, dtype=torch.float64, device=dev)
        self.a[1:-1] = self.rf[1:-1] / self.dzn
        self.vol = self.rc * self.dz

    def div(self, u, v, w):
        d = (u - u.roll(1, 2)) / self.dx
        d += (v - v.roll(1, 1)) / self.dy
        f = self.rf[:, None, None] * w
        f[0].zero_()
        f[-1].zero_()
        d += (f[1:] - f[:-1]) / self.vol[:, None, None]
        return d

    def thomas(self, lam, d):
        """(A[k] p[k-1] - (A[k]+A[k+1]) p[k] + A[k+1] p[k+1])/vol[k] + lam p[k] = d[k], in place."""
        a = self.a.tolist()
        vol = self.vol.tolist()
        g = torch.empty((self.nz,) + tuple(lam.shape), dtype=torch.float64, device=d.device)
        for k in range(self.nz):
            e = lam * vol[k] - (a[k] + a[k + 1])
            d[k] *= vol[k]
            if k:
                e -= a[k] * a[k] * g[k - 1]
                d[k] -= d[k - 1] * (a[k] * g[k - 1])
            g[k] = 1.0 / e
            if k == 0:
                self._pin(lam, g, d)
        d[-1] *= g[-1]
        for k in range(self.nz - 2, -1, -1):
            d[k] = (d[k] - a[k + 1] * d[k + 1]) * g[k]
        return d

    @staticmethod
    def _pin(lam, g, d):
        if lam.dim() == 2 and float(lam[0, 0]) == 0.0:
            g[0, 0, 0] = 0.0
            d[0, 0, 0] = 0.0


def _exact_fft(g, u, v, w, phi):
    op = _Op(g)
    u, v, w = u.double(), v.double(), w.double()
    dev = u.device
    kx = torch.arange(g.nx // 2 + 1, device=dev, dtype=torch.float64)
    ky = torch.arange(g.ny, device=dev, dtype=torch.float64)
    sx, sy = torch.sin(math.pi * kx / g.nx), torch.sin(math.pi * ky / g.ny)
    lam = -4 * sx[None, :] ** 2 / g.dx ** 2 - 4 * sy[:, None] ** 2 / g.dy ** 2
    lam[0, 0] = 0.0
    p = op.thomas(lam, torch.fft.rfft2(op.div(u, v, w)))
    ex = torch.complex(-2 * sx ** 2, torch.sin(2 * math.pi * kx / g.nx)) / g.dx
    ey = torch.complex(-2 * sy ** 2, torch.sin(2 * math.pi * ky / g.ny)) / g.dy
    back = lambda s: torch.fft.irfft2(s, s=(g.ny, g.nx))  # noqa: E731
    u -= back(p * ex[None, None, :])
    v -= back(p * ey[None, :, None])
    if g.nz > 1:
        w[1:-1] -= back((p[1:] - p[:-1]) / op.dzn[:, None, None])
    w[0].zero_()
    w[-1].zero_()
    return [u, v, w] + ([back(p)] if phi else [])


def _exact_krylov(g, u, v, w):
    """BiCGStab from zero with the vertical lines as preconditioner, a fixed number of iterations."""
    op = _Op(g)
    u, v, w = u.double(), v.double(), w.double()
    a, vol = op.a[:, None, None], op.vol[:, None, None]

    def lap(x):
        y = (x.roll(-1, 2) - 2 * x + x.roll(1, 2)) / g.dx ** 2
        y += (x.roll(-1, 1) - 2 * x + x.roll(1, 1)) / g.dy ** 2
        if g.nz > 1:
            f = a[1:-1] * (x[1:] - x[:-1])
            y[:-1] += f / vol[:-1]
            y[1:] -= f / vol[1:]
        return y

    hdiag = torch.full((1, 1), -2 / g.dx ** 2 - 2 / g.dy ** 2, dtype=torch.float64, device=u.device)
    line = lambda x: op.thomas(hdiag, x.clone())  # noqa: E731
    dot = lambda x, y: float((x * y).sum())  # noqa: E731
    b = op.div(u, v, w)
    r, p, q = b.clone(), b.clone(), None
    x = torch.zeros_like(b)
    rho, beta, omega = dot(b, b), 0.0, 1.0
    for it in range(KRYLOV_ITERS):
        if it:
            p = r + beta * (p - omega * q)
        ph = line(p)
        q = lap(ph)
        alpha = rho / dot(b, q)
        r -= alpha * q
        sh = line(r)
        t = lap(sh)
        omega = dot(t, r) / dot(t, t)
        x += alpha * ph + omega * sh
        r -= omega * t
        new = dot(b, r)
        beta, rho = (new / rho) * (alpha / omega), new
    x -= x[0].mean()
    u -= (x.roll(-1, 2) - x) / g.dx
    v -= (x.roll(-1, 1) - x) / g.dy
    if g.nz > 1:
        w[1:-1] -= (x[1:] - x[:-1]) / op.dzn[:, None, None]
    w[0].zero_()
    w[-1].zero_()
    return u, v, w, x


def exact(case, seed):
    grids, fields = _inputs(case, seed)
    if case["kind"] == "krylov":
        u, v, w, phi = _exact_krylov(grids[0], *fields[0])
        return {"u": u, "v": v, "w": w, "phi": phi if case["phi"] else None, "iterations": None}
    got = [_exact_fft(g, *f, bool(case.get("phi"))) for g, f in zip(grids, fields)]
    return got if case["kind"] == "batch" else got[0]
