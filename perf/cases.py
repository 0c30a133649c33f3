"""The work that users of this library have it do, as timed cases.

Each case is one call (or the fixed handful of calls of one time step) through
paper_2509_19061_gb300.api, at the sizes of the repository's configurations,
tests and benchmark.  The inputs are the synthetic ones of
paper_2509_19061_gb300/inputs.py (sinkers, multi-sinkers, layers), formed on
the device from the seed; `exact` restates the maps in plain FP64 torch.
"""
import math

import numpy as np
import torch

from paper_2509_19061_gb300 import api, inputs

DEV = "cuda"


def listed():
    return [
        # the smallest configuration, plain FP64: a 64 x 64 sinker, ten RAS sweeps on 8 x 8 tiles (latency of a call)
        dict(name="sinker64_f64_ras", kind="smooth", dtype="f64", nx=64, ny=64, lx=1.0, ly=1.0, material="sinker",
             pressure=False, variant="ras", sweeps=10, ti=8, tj=8, k=2, overlap=1),
        # FP64 smoothing at 1024^2, contrast 1e4: the smoother comparison's RAS schedule, 100 sweeps, L2-resident
        dict(name="sinker1024_f64_ras", kind="smooth", dtype="f64", nx=1024, ny=1024, lx=1.0, ly=1.0,
             material="sinker", pressure=False, variant="ras", sweeps=100, ti=32, tj=32, k=4, overlap=3),
        # the benchmark's step: new viscosity and force, 100 RAS sweeps from rest and the energy norm at 8192^2, FP32
        dict(name="layered8192_f32_step", kind="step", dtype="f32", nx=8192, ny=8192, lx=1.0, ly=1.0,
             material="layers", sweeps=100, ti=48, tj=64, k=8, overlap=7),
        # 20 fused Jacobi sweeps of a velocity with a pressure on a ragged grid of oblong cells, FP32
        dict(name="ragged_f32_fused", kind="smooth", dtype="f32", nx=4001, ny=2999, lx=1.3, ly=0.9, material="multi",
             pressure=True, variant="fused", sweeps=20, ti=0, tj=0, k=1, overlap=0),
        # 20 red-black Gauss-Seidel sweeps at 2000^2, the comparison smoother at the paper's smallest timed size
        dict(name="rbgs2000_f32", kind="smooth", dtype="f32", nx=2000, ny=2000, lx=1.0, ly=1.0, material="layers",
             pressure=False, variant="rbgs", sweeps=20, ti=0, tj=0, k=1, overlap=0),
        # a solver's own check of its state: M v + G p and the energy norm in FP64 at 2000^2
        dict(name="residual2000_f64", kind="residual", dtype="f64", nx=2000, ny=2000, lx=1.0, ly=1.0,
             material="layers"),
        # one time step of a velocity solver: new viscosity and force, then eight V-cycle-preconditioned CG
        # iterations (FP32 sweeps inside FP64), hierarchy and graph rebuilt with the viscosity
        dict(name="newstep1024_f64_f32", kind="solve", dtype="f64", inner="f32", nx=1024, ny=1024, material="multi",
             new_eta=True, cycles=8, ti=48, tj=32, k=8, overlap=7),
        # the time-to-residual workload, 4096^2 multi-sinker: six CG iterations of a solve whose hierarchy is kept
        dict(name="solve4096_f64_f32", kind="solve", dtype="f64", inner="f32", nx=4096, ny=4096, material="multi",
             new_eta=False, cycles=6, ti=48, tj=64, k=8, overlap=7),
        # the inexact Uzawa Stokes solve with viscosity continuation (five stages of three cycles) at 512^2
        dict(name="uzawa512_f64_f32", kind="uzawa", dtype="f64", inner="f32", nx=512, ny=512, material="sinker",
             cycles=15, interval=3, vel_its=2, ti=32, tj=32, k=4, overlap=3),
        # the batched workload: 256 sinkers of 64^2 to 1024^2 cells smoothed together, 20 FP32 RAS sweeps
        dict(name="batch256_f32_smooth", kind="batch_smooth", dtype="f32", count=256, sizes=5, sweeps=20, ti=48,
             tj=64, k=8, overlap=7),
        # 64 of them solved together: four FP64 CG iterations around the batched FP32 V-cycle
        dict(name="batch64_f64_f32_solve", kind="batch_solve", dtype="f64", inner="f32", count=64, sizes=5, cycles=4,
             ti=48, tj=64, k=8, overlap=7),
        # the 3D operator: eight RAS sweeps on 30 x 6 x 6 tiles of the 384^3 layered sinker, FP32
        dict(name="box384_f32_ras3d", kind="smooth3d", dtype="f32", nx=384, ny=384, nz=384, variant="ras", sweeps=8,
             ti=30, tj=6, tk=6, k=4, overlap=0),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["smooth"] * 6 + ["step", "residual", "solve", "solve", "uzawa", "batch_smooth", "batch_solve",
                                        "smooth3d", "smooth3d"])
    dtype = rng.choice(["f32", "f32", "f64"])
    material = rng.choice(["sinker", "layers", "multi"])
    if kind in ("smooth", "step", "residual"):
        top = 6000 if dtype == "f32" else 2500
        nx = _log_int(rng, 40, top)
        ny = max(30, min(top, int(nx * rng.uniform(0.6, 1.6))))
        lx = 1.0
        ly = rng.choice([ny / nx, round(rng.uniform(0.7, 1.4), 3)])
        case = dict(kind=kind, dtype=dtype, nx=nx, ny=ny, lx=lx, ly=ly, material=material)
        if kind == "residual":
            return case
        scheds = [(32, 32, 4, 3), (48, 64, 8, 7), (48, 32, 8, 7), (56, 32, 4, 3), (16, 16, 2, 1), (32, 32, 8, 0),
                  (62, 56, 8, 0), (56, 32, 8, 0)]
        if dtype == "f64":
            scheds = [(32, 32, 4, 3), (32, 32, 2, 1), (16, 16, 8, 0), (16, 16, 2, 1), (24, 24, 8, 7), (32, 32, 8, 0)]
        ti, tj, k, o = rng.choice(scheds)
        if kind == "step":
            return dict(case, sweeps=rng.randint(8, 50), ti=ti, tj=tj, k=k, overlap=o)
        variant = rng.choice(["ras", "ras", "ras", "jacobi", "fused", "blocked", "rbgs"])
        return dict(case, pressure=rng.random() < 0.5, variant=variant, sweeps=rng.randint(1, 30), ti=ti, tj=tj, k=k,
                    overlap=o)
    if kind in ("solve", "uzawa"):
        # sides that halve to a coarsest level of at most 16 cells
        n = 16 << rng.randint(2, 6 if kind == "solve" else 5)
        nx, ny = n, n // 4 * rng.choice([3, 4, 4])
        inner = rng.choice(["f32", "f32", "f64"])
        ti, tj, k, o = rng.choice([(32, 32, 4, 3), (16, 16, 8, 0)] +
                                  ([(48, 32, 8, 7), (48, 64, 8, 7)] if inner == "f32" else [(24, 24, 4, 3)]))
        if kind == "solve":
            return dict(kind=kind, dtype="f64", inner=inner, nx=nx, ny=ny, material=material,
                        new_eta=rng.random() < 0.5, cycles=rng.randint(2, 6), ti=ti, tj=tj, k=k, overlap=o)
        return dict(kind=kind, dtype="f64", inner=inner, nx=nx, ny=ny, material="sinker", cycles=rng.randint(4, 10),
                    interval=rng.choice([0, 2]), vel_its=rng.randint(1, 2), ti=ti, tj=tj, k=k, overlap=o)
    if kind in ("batch_smooth", "batch_solve"):
        ti, tj, k, o = rng.choice([(48, 64, 8, 7), (32, 32, 4, 3), (56, 32, 8, 0)])
        case = dict(kind=kind, count=_log_int(rng, 4, 200 if kind == "batch_smooth" else 48),
                    sizes=rng.randrange(1000), ti=ti, tj=tj, k=k, overlap=o)
        if kind == "batch_smooth":
            return dict(case, dtype="f32", sweeps=rng.randint(4, 30))
        return dict(case, dtype="f64", inner="f32", cycles=rng.randint(2, 4))
    n = _log_int(rng, 24, 320 if dtype == "f32" else 160)
    ny, nz = (max(16, int(n * rng.uniform(0.7, 1.1))) for _ in range(2))
    variant = rng.choice(["ras", "ras", "fused"])
    ti, tj, tk, k, o = rng.choice([(30, 6, 6, 4, 0), (8, 8, 8, 2, 1), (28, 4, 4, 2, 1), (8, 8, 8, 4, 0)] +
                                  ([(30, 14, 6, 8, 0), (28, 8, 4, 2, 1)] if dtype == "f32" else []))
    return dict(kind="smooth3d", dtype=dtype, nx=n, ny=ny, nz=nz, variant=variant, sweeps=rng.randint(2, 8), ti=ti,
                tj=tj, tk=tk, k=k, overlap=o)


# --------------------------------------------------------------------------
# inputs, on the device (FP64, natural staggered shapes)
# --------------------------------------------------------------------------
def _arange(n, h, at):
    return (torch.arange(n, dtype=torch.float64, device=DEV) + at) * h


def _materials(c, seed):
    """eta_c, eta_n, fx, fy of a case (inputs.py's generators, geometry drawn from the seed)."""
    nx, ny, lx, ly = c["nx"], c["ny"], c.get("lx", 1.0), c.get("ly", c["ny"] / c["nx"])
    hx, hy = lx / nx, ly / ny
    rng = np.random.default_rng([seed, 11])
    at = {"c": (_arange(nx, hx, 0.5), _arange(ny, hy, 0.5)), "n": (_arange(nx + 1, hx, 0.0), _arange(ny + 1, hy, 0.0)),
          "r": (_arange(nx, hx, 0.5), _arange(ny + 1, hy, 0.0))}
    f = {"c": torch.ones((ny, nx), dtype=torch.float64, device=DEV),
         "n": torch.ones((ny + 1, nx + 1), dtype=torch.float64, device=DEV),
         "r": torch.ones((ny + 1, nx), dtype=torch.float64, device=DEV)}

    def disc(cx, cy, r, eta, rho):
        for key, val in (("c", eta), ("n", eta), ("r", rho)):
            xs, ys = at[key]
            i0, i1 = (int(v) for v in torch.searchsorted(xs, xs.new_tensor([cx - r, cx + r])).tolist())
            j0, j1 = (int(v) for v in torch.searchsorted(ys, ys.new_tensor([cy - r, cy + r])).tolist())
            if i0 >= i1 or j0 >= j1:
                continue
            m = (xs[None, i0:i1] - cx) ** 2 + (ys[j0:j1, None] - cy) ** 2 < r * r
            f[key][j0:j1, i0:i1].masked_fill_(m, val)

    side = min(lx, ly)
    if c["material"] == "layers":
        for q in range(10):
            eta = 10.0 ** rng.uniform(-3.0, 3.0)
            for key in ("c", "n"):
                ys = at[key][1]
                f[key][ys >= q * ly / 10] = eta
        disc(lx * rng.uniform(0.4, 0.6), ly * rng.uniform(0.4, 0.6), 0.1 * side, 1e3, 2.0)
    elif c["material"] == "multi":
        for _ in range(20):
            r = rng.uniform(0.02, 0.08)
            cx, cy = rng.uniform(r, 1.0 - r), rng.uniform(r, 1.0 - r)
            disc(lx * cx, ly * cy, r * side, 10.0 ** rng.uniform(-3.0, 3.0), rng.uniform(0.9, 1.1))
    else:
        disc(lx * rng.uniform(0.4, 0.6), ly * rng.uniform(0.4, 0.6), side * rng.uniform(0.08, 0.15), 1e4, 2.0)
    fx = torch.zeros((ny, nx + 1), dtype=torch.float64, device=DEV)
    fy = f["r"]
    fy[0] = 0.0
    fy[ny] = 0.0
    return f["c"], f["n"], fx, fy


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed) * 7 + 3)


def _velocity(c, seed):
    """A smooth flow plus small-scale noise, zero on the walls: what a smoother is handed."""
    nx, ny = c["nx"], c["ny"]
    g = _gen(seed)
    vx = 1e-3 * torch.randn((ny, nx + 1), dtype=torch.float64, device=DEV, generator=g)
    vy = 1e-3 * torch.randn((ny + 1, nx), dtype=torch.float64, device=DEV, generator=g)
    x, y = _arange(nx + 1, math.pi / nx, 0.0), _arange(ny + 1, math.pi / ny, 0.0)
    xc, yc = _arange(nx, math.pi / nx, 0.5), _arange(ny, math.pi / ny, 0.5)
    vx += 1e-2 * torch.sin(x)[None, :] * torch.cos(yc)[:, None]
    vy -= 1e-2 * torch.cos(xc)[None, :] * torch.sin(y)[:, None]
    vx[:, 0] = vx[:, nx] = 0.0
    vy[0] = vy[ny] = 0.0
    return vx, vy


def _pressure(c, seed):
    return torch.randn((c["ny"], c["nx"]), dtype=torch.float64, device=DEV, generator=_gen(seed + 1))


def _put(ctx, a):
    """A natural-shape field in the context's pitched layout and dtype."""
    t = ctx.field()
    t[tuple(slice(0, s) for s in a.shape)] = a.to(t.dtype)
    return t


def _materials3d(c, seed):
    n = (c["nx"], c["ny"], c["nz"])
    rng = np.random.default_rng([seed, 13])
    layer = torch.tensor(10.0 ** rng.uniform(-3.0, 3.0, size=10), device=DEV)
    centre = rng.uniform(0.4, 0.6, size=3)

    def sample(stag, inside, back):
        axes = [_arange(m + s, 1.0 / m, 0.0 if s else 0.5) for m, s in zip(n, stag)]
        x, y, z = axes[0][None, None, :], axes[1][None, :, None], axes[2][:, None, None]
        ball = (x - centre[0]) ** 2 + (y - centre[1]) ** 2 + (z - centre[2]) ** 2 < 0.01
        b = layer[(z * 10).long().clamp(0, 9)] if back is None else torch.full_like(z, back)
        return torch.where(ball, torch.tensor(inside, dtype=torch.float64, device=DEV), b)

    eta = [sample(s, 1e3, None) for s in ((0, 0, 0), (1, 1, 0), (1, 0, 1), (0, 1, 1))]
    fz = sample((0, 0, 1), 2.0, 1.0).contiguous()
    fz[0] = 0.0
    fz[-1] = 0.0
    nx, ny, nz = n
    zero = dict(dtype=torch.float64, device=DEV)
    f = [torch.zeros((nz, ny, nx + 1), **zero), torch.zeros((nz, ny + 1, nx), **zero), fz]
    g = _gen(seed)
    v = [1e-3 * torch.randn(a.shape, generator=g, **zero) for a in f]
    v[0][:, :, 0] = v[0][:, :, -1] = 0.0
    v[1][:, 0] = v[1][:, -1] = 0.0
    v[2][0] = v[2][-1] = 0.0
    return eta, f, v


def _specs(c, seed):
    """Instance sides fixed by the case, contrast and geometry by the seed (inputs.batch_specs)."""
    side = [s.n for s in inputs.batch_specs(seed=c["sizes"], count=c["count"])]
    return [(n, s) for n, s in zip(side, inputs.batch_specs(seed=seed, count=c["count"]))]


def _batch_materials(n, s):
    x, xn = _arange(n, 1.0 / n, 0.5), _arange(n + 1, 1.0 / n, 0.0)

    def disc(xs, ys, val):
        m = (xs[None, :] - s.cx) ** 2 + (ys[:, None] - s.cy) ** 2 < s.radius ** 2
        return torch.where(m, torch.tensor(val, dtype=torch.float64, device=DEV), 1.0)

    fy = disc(x, xn, 2.0)
    fy[0] = fy[n] = 0.0
    return disc(x, x, s.contrast), disc(xn, xn, s.contrast), torch.zeros((n, n + 1), dtype=torch.float64, device=DEV), fy


# --------------------------------------------------------------------------
# the calls
# --------------------------------------------------------------------------
def _ras(c):
    return dict(tile=(c["ti"], c["tj"]), k=c["k"], overlap=c["overlap"], seed=1)


def prepare(case, seed):
    c, kind = case, case["kind"]
    if kind == "smooth3d":
        eta, f, v = _materials3d(c, seed)
        ctx = api.Stokes3DContext(c["nx"], c["ny"], c["nz"], 1.0, 1.0, 1.0, c["dtype"])
        api.stokes3d_set_viscosity(ctx.ctx, *[_put(ctx, a) for a in eta])
        api.stokes3d_set_rhs(ctx.ctx, *[_put(ctx, a) for a in f])
        kw = dict(variant=c["variant"], sweeps=c["sweeps"])
        if c["variant"] == "ras":
            kw.update(tile=(c["ti"], c["tj"], c["tk"]), k=c["k"], overlap=c["overlap"], seed=1)
        state = dict(c=c, ctx=ctx, v=[_put(ctx, a) for a in v], kw=kw)
    elif kind in ("batch_smooth", "batch_solve"):
        specs = _specs(c, seed)
        sides = [n for n, _ in specs]
        ctx = api.BatchContext(sides, sides, dtype=c["dtype"])
        slabs = [ctx.slab() for _ in range(4)]
        for i, (n, s) in enumerate(specs):
            for slab, a in zip(slabs, _batch_materials(n, s)):
                ctx.view(slab, i)[:a.shape[0], :a.shape[1]] = a.to(slab.dtype)
        api.stokes_batch_set_viscosity(ctx.b, slabs[0], slabs[1])
        api.stokes_batch_set_rhs(ctx.b, slabs[2], slabs[3])
        state = dict(c=c, ctx=ctx, vx=ctx.slab(), vy=ctx.slab())
    else:
        ec, en, fx, fy = _materials(c, seed)
        ctx = api.StokesContext(c["nx"], c["ny"], c.get("lx", 1.0), c.get("ly", c["ny"] / c["nx"]), c["dtype"])
        eta, f = (_put(ctx, ec), _put(ctx, en)), (_put(ctx, fx), _put(ctx, fy))
        ctx.set_viscosity_dev(*eta)
        ctx.set_rhs_dev(*f)
        state = dict(c=c, ctx=ctx, eta=eta, f=f, p=None)
        if kind in ("smooth", "residual"):
            vx, vy = _velocity(c, seed)
            state.update(vx=_put(ctx, vx), vy=_put(ctx, vy))
        else:
            state.update(vx=ctx.field(), vy=ctx.field())
        if c.get("pressure") or kind == "residual":
            state["p"] = _put(ctx, _pressure(c, seed))
        if kind == "uzawa":
            state["p"] = ctx.field()
    torch.cuda.synchronize()
    return state


def run(state):
    c, ctx = state["c"], state["ctx"]
    kind = c["kind"]
    if kind == "smooth3d":
        ctx.smooth(*state["v"], None, **state["kw"])
        return list(state["v"])
    vx, vy = state["vx"], state["vy"]
    if kind == "smooth":
        ctx.smooth(vx, vy, state["p"], variant=c["variant"], sweeps=c["sweeps"], **_ras(c))
        return vx, vy
    if kind == "residual":
        ox, oy = ctx.apply(vx, vy, state["p"])
        return ox, oy, np.array(ctx.energy(vx, vy, state["p"]))
    if kind == "batch_smooth":
        ctx.smooth(vx, vy, None, variant="ras", sweeps=c["sweeps"], **_ras(c))
        return vx, vy
    # the others start from rest
    vx.zero_()
    vy.zero_()
    if kind == "step":
        ctx.set_viscosity_dev(*state["eta"])
        ctx.set_rhs_dev(*state["f"])
        ctx.smooth(vx, vy, None, variant="ras", sweeps=c["sweeps"], **_ras(c))
        return vx, vy, np.array(ctx.energy(vx, vy, None))
    kw = dict(_ras(c), variant="ras", nu_max=40, inner=c["inner"], krylov=True)
    if kind == "solve":
        if c["new_eta"]:
            ctx.set_viscosity_dev(*state["eta"])
            ctx.set_rhs_dev(*state["f"])
        ctx.vcycle(vx, vy, None, tol=1e-12, max_cycles=c["cycles"], **kw)
        return vx, vy
    if kind == "batch_solve":
        ctx.solve(vx, vy, None, tol=1e-12, max_cycles=c["cycles"], **kw)
        return vx, vy
    _, hist, _, _ = ctx.uzawa(vx, vy, state["p"], cycles=c["cycles"], theta_interval=c["interval"],
                              vel_its=c["vel_its"], **kw)
    return vx, vy, state["p"], hist


def work(case):
    """Bytes: every input field read once, every output field written once.  Flops: 24 per 2D cell and sweep (51 in
    3D: six stresses, three components), the stencil's algorithmic count; a V-cycle of a solve counts its finest
    level's ten sweeps, residual and operator, the coarser levels a third of that."""
    c, kind = case, case["kind"]
    es = 8 if c["dtype"] == "f64" else 4
    if kind == "smooth3d":
        cells = c["nx"] * c["ny"] * c["nz"]
        return dict(bytes=13.0 * es * cells, flops=51.0 * cells * c["sweeps"])
    if kind in ("batch_smooth", "batch_solve"):
        cells = sum(s.n ** 2 for s in inputs.batch_specs(seed=c["sizes"], count=c["count"]))
    else:
        cells = c["nx"] * c["ny"]
    sweep = 24.0 * cells
    if kind in ("smooth", "batch_smooth"):
        words = 8 + (1 if c.get("pressure") else 0)
        return dict(bytes=float(words * es * cells), flops=sweep * c["sweeps"])
    if kind == "step":
        return dict(bytes=6.0 * es * cells, flops=sweep * (c["sweeps"] + 2))
    if kind == "residual":
        return dict(bytes=9.0 * es * cells, flops=2 * sweep)
    cycles = c["cycles"] * c.get("vel_its", 1)
    return dict(bytes=(7.0 if kind == "uzawa" else 6.0) * es * cells, flops=sweep * cycles * 12 * 4 / 3)


# --------------------------------------------------------------------------
# the same maps in FP64 torch
# --------------------------------------------------------------------------
def _at(a, c):
    """The value the call gets: the FP64 input rounded to the case's dtype."""
    return a.to(torch.float32).double() if c["dtype"] == "f32" else a


def _diff(a, dim):
    return a.diff(dim=dim)


class _Op2:
    """The operator on natural staggered arrays; eta_n counts on interior nodes only."""

    def __init__(self, c, ec, en):
        self.hx, self.hy = c.get("lx", 1.0) / c["nx"], c.get("ly", c["ny"] / c["nx"]) / c["ny"]
        self.ec = ec
        self.en = en.clone()
        self.en[0] = self.en[-1] = 0.0
        self.en[:, 0] = self.en[:, -1] = 0.0
        hx2, hy2 = self.hx ** 2, self.hy ** 2
        self.dx = -(2 * (ec[:, 1:] + ec[:, :-1]) / hx2 + (self.en[1:, 1:-1] + self.en[:-1, 1:-1]) / hy2)
        self.dy = -(2 * (ec[1:] + ec[:-1]) / hy2 + (self.en[1:-1, 1:] + self.en[1:-1, :-1]) / hx2)

    def shear(self, vx, vy):
        s = torch.zeros_like(self.en)
        s[1:-1, 1:-1] = self.en[1:-1, 1:-1] * (_diff(vx[:, 1:-1], 0) / self.hy + _diff(vy[1:-1], 1) / self.hx)
        return s

    def mx(self, vx, s):
        return _diff(2 * self.ec * _diff(vx, 1) / self.hx, 1) / self.hx + _diff(s[:, 1:-1], 0) / self.hy

    def my(self, vy, s):
        return _diff(2 * self.ec * _diff(vy, 0) / self.hy, 0) / self.hy + _diff(s[1:-1], 1) / self.hx


def _padded(ctx_pitch, ny, a):
    out = torch.zeros((ny + 1, ctx_pitch), dtype=torch.float64, device=DEV)
    out[:a.shape[0], :a.shape[1]] = a
    return out


def _pitch(nx):
    return (nx + 1 + 31) // 32 * 32


def _jacobi(op, bx, by, vx, vy, sweeps, omega=0.3):
    for _ in range(sweeps):
        s = op.shear(vx, vy)
        ux = omega * (bx[:, 1:-1] - op.mx(vx, s)) / op.dx
        uy = omega * (by[1:-1] - op.my(vy, s)) / op.dy
        vx[:, 1:-1] += ux
        vy[1:-1] += uy


def _rbgs(op, bx, by, vx, vy, sweeps, omega=0.3):
    def parity(a, j0, i0):
        j = torch.arange(j0, j0 + a.shape[0], device=DEV)
        i = torch.arange(i0, i0 + a.shape[1], device=DEV)
        return (j[:, None] + i[None, :]) % 2
    px, py = parity(vx[:, 1:-1], 0, 1), parity(vy[1:-1], 1, 0)
    for _ in range(sweeps):
        for colour in (0, 1):
            u = omega * (bx[:, 1:-1] - op.mx(vx, op.shear(vx, vy))) / op.dx
            vx[:, 1:-1] += u * (px == colour)
        for colour in (0, 1):
            u = omega * (by[1:-1] - op.my(vy, op.shear(vx, vy))) / op.dy
            vy[1:-1] += u * (py == colour)


def _splitmix(seed, n):
    m = (1 << 64) - 1
    z = (seed + (n + 1) * 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _windows(n, t, s, h):
    """Tiles of [0, n) cut at s + m t: their first cells, ends, and the indices of their windows (h cells around)."""
    cuts = [0] + list(range(s if s > 0 else t, n, t)) + [n]
    lo = torch.tensor(cuts[:-1], device=DEV)
    hi = torch.tensor(cuts[1:], device=DEV)
    return lo, hi, lo[:, None] - h + torch.arange(t + 2 * h, device=DEV)[None, :]


def _tiled(dims, sizes, shifts, overlap, sweeps, fields, v, update):
    """RAS: every tile's window (cells grown by overlap + 1) runs `sweeps` local sweeps from the snapshot and writes
    back its own cells.  dims: cells per axis in array order; fields and v: arrays of dims + 1, zero outside their
    extent; update(windows of fields, windows of v): the increments at every window cell."""
    nd = len(dims)
    w = [_windows(n, t, s, overlap + 1) for n, t, s in zip(dims, sizes, shifts)]

    def shape(t, axis):  # axis's tile and cell dimensions among all
        view = [1] * (2 * nd)
        view[axis] = t.shape[0]
        if t.dim() == 2:
            view[nd + axis] = t.shape[1]
        return t.reshape(view)

    inside, grown, owned, index = True, True, True, []
    for a, (n, (lo, hi, ix)) in enumerate(zip(dims, w)):
        inside = inside & shape((ix >= 0) & (ix <= n), a)
        grown = grown & shape((ix >= lo[:, None] - overlap) & (ix < hi[:, None] + overlap), a)
        owned = owned & shape((ix >= lo[:, None]) & (ix < hi[:, None]), a)
        index.append(shape(ix.clamp(0, n), a))
    take = lambda f: f[tuple(index)] * inside  # noqa: E731
    fw, vw = [take(f) for f in fields], [take(x) for x in v]
    for _ in range(sweeps):
        for x, u in zip(vw, update(fw, vw)):
            x += u * grown
    full = torch.broadcast_tensors(owned, vw[0])[0]
    at = tuple(torch.broadcast_to(i, full.shape)[full] for i in index)
    for x, new in zip(v, vw):
        x[at] = new[full]


def _east(a, axis):
    return torch.roll(a, -1, axis)


def _west(a, axis):
    return torch.roll(a, 1, axis)


def _ras2(c, op, bx, by, vx, vy, omega=0.3):
    nx, ny = c["nx"], c["ny"]
    full = lambda a: torch.nn.functional.pad(a, (0, nx + 1 - a.shape[1], 0, ny + 1 - a.shape[0]))  # noqa: E731
    wx = torch.zeros((ny + 1, nx + 1), dtype=torch.float64, device=DEV)
    wy = wx.clone()
    wx[:ny, 1:nx] = omega / op.dx
    wy[1:ny, :nx] = omega / op.dy
    fields = [full(op.ec), op.en, full(bx), full(by), wx, wy]
    v = [full(vx), full(vy)]

    def update(f, u):
        ec, en, b0, b1, w0, w1 = f
        x, y = u
        txx = 2 * ec * (_east(x, -1) - x) / op.hx
        tyy = 2 * ec * (_east(y, -2) - y) / op.hy
        s = en * ((x - _west(x, -2)) / op.hy + (y - _west(y, -1)) / op.hx)
        mx = (txx - _west(txx, -1)) / op.hx + (_east(s, -2) - s) / op.hy
        my = (_east(s, -1) - s) / op.hx + (tyy - _west(tyy, -2)) / op.hy
        return w0 * (b0 - mx), w1 * (b1 - my)

    done, t = 0, 0
    while done < c["sweeps"]:
        ks = min(c["k"], c["sweeps"] - done)
        si, sj = _splitmix(1, 2 * t) % c["ti"], _splitmix(1, 2 * t + 1) % c["tj"]
        _tiled((ny, nx), (c["tj"], c["ti"]), (sj, si), c["overlap"], ks, fields, v, update)
        done, t = done + ks, t + 1
    vx.copy_(v[0][:ny, :nx + 1])
    vy.copy_(v[1][:ny + 1, :nx])


def _energy(op, bx, by, fx, fy, vx, vy):
    s = op.shear(vx, vy)
    rx, ry = bx[:, 1:-1] - op.mx(vx, s), by[1:-1] - op.my(vy, s)
    d = _diff(vx, 1) / op.hx + _diff(vy, 0) / op.hy
    w = 2 / op.hx ** 2 + 2 / op.hy ** 2
    return torch.stack([-(rx ** 2 / op.dx).sum() - (ry ** 2 / op.dy).sum(), (d ** 2 * op.ec / w).sum(),
                        -(fx[:, 1:-1] ** 2 / op.dx).sum() - (fy[1:-1] ** 2 / op.dy).sum()]).cpu().numpy()


def _exact_3d(c, seed):
    (ec, exy, exz, eyz), f, v = (tuple(_at(a, c) for a in part) for part in _materials3d(c, seed))
    nx, ny, nz = c["nx"], c["ny"], c["nz"]
    h = (1.0 / nx, 1.0 / ny, 1.0 / nz)
    full = lambda a: torch.nn.functional.pad(  # noqa: E731
        a, (0, nx + 1 - a.shape[2], 0, ny + 1 - a.shape[1], 0, nz + 1 - a.shape[0]))
    exy, exz, eyz = exy.clone(), exz.clone(), eyz.clone()
    # no shear stress on the edges that lie in the walls
    exy[:, 0] = exy[:, -1] = 0.0
    exy[:, :, 0] = exy[:, :, -1] = 0.0
    exz[0] = exz[-1] = 0.0
    exz[:, :, 0] = exz[:, :, -1] = 0.0
    eyz[0] = eyz[-1] = 0.0
    eyz[:, 0] = eyz[:, -1] = 0.0
    ec, exy, exz, eyz = (full(a) for a in (ec, exy, exz, eyz))
    edge = {(0, 1): exy, (0, 2): exz, (1, 2): eyz}
    ax = (-1, -2, -3)  # the array axis of x, y, z
    weights = []
    for a in range(3):
        d = -2 * (ec + _west(ec, ax[a])) / h[a] ** 2
        for o in range(3):
            if o != a:
                e = edge[tuple(sorted((a, o)))]
                d = d - (_east(e, ax[o]) + e) / h[o] ** 2
        unknown = torch.zeros_like(ec, dtype=torch.bool)
        ext = [slice(0, nz), slice(0, ny), slice(0, nx)]
        ext[2 - a] = slice(1, (nx, ny, nz)[a])
        unknown[tuple(ext)] = True
        weights.append(torch.where(unknown, 0.3 / torch.where(unknown, d, 1.0), 0.0))
        del d, unknown
    vv = [full(a) for a in v]
    fields = [ec, exy, exz, eyz] + [full(a) for a in f] + weights

    def update(fs, u):
        e = {(0, 1): fs[1], (0, 2): fs[2], (1, 2): fs[3]}
        shear = {(a, o): e[a, o] * ((u[a] - _west(u[a], ax[o])) / h[o] + (u[o] - _west(u[o], ax[a])) / h[a])
                 for a, o in e}
        out = []
        for a in range(3):
            t = 2 * fs[0] * (_east(u[a], ax[a]) - u[a]) / h[a]
            m = (t - _west(t, ax[a])) / h[a]
            for o in range(3):
                if o != a:
                    s = shear[tuple(sorted((a, o)))]
                    m = m + (_east(s, ax[o]) - s) / h[o]
            out.append(fs[7 + a] * (fs[4 + a] - m))
        return out

    if c["variant"] == "ras" and c["overlap"] < c["k"] - 1:
        done, t = 0, 0
        while done < c["sweeps"]:
            ks = min(c["k"], c["sweeps"] - done)
            s = [_splitmix(1, 3 * t + q) % c[key] for q, key in enumerate(("ti", "tj", "tk"))]
            _tiled((nz, ny, nx), (c["tk"], c["tj"], c["ti"]), (s[2], s[1], s[0]), c["overlap"], ks, fields, vv, update)
            done, t = done + ks, t + 1
    else:
        for _ in range(c["sweeps"]):
            for x, u in zip(vv, update(fields, vv)):
                x += u
    out = []
    for x in vv:
        o = torch.zeros((nz + 1, ny + 1, _pitch(nx)), dtype=torch.float64, device=DEV)
        o[:, :, :nx + 1] = x
        out.append(o)
    return out


def exact(case, seed):
    c, kind = case, case["kind"]
    if kind in ("solve", "uzawa", "batch_solve"):
        return None  # iterates of an FP32-preconditioned iteration, not of a map stated in 64 bits
    if kind == "smooth3d":
        return _exact_3d(c, seed)
    if kind == "batch_smooth":
        if c["overlap"] < c["k"] - 1:
            return None  # hundreds of tilings of uneven grids
        outs = [[], []]
        for n, s in _specs(c, seed):
            cc = dict(c, nx=n, ny=n)
            ec, en, fx, fy = (_at(a, c) for a in _batch_materials(n, s))
            vx, vy = torch.zeros_like(fx), torch.zeros_like(fy)
            _jacobi(_Op2(cc, ec, en), fx, fy, vx, vy, c["sweeps"])
            for o, a in zip(outs, (vx, vy)):
                part = _padded(_pitch(n), n, a).reshape(-1)
                # the slab's instances start at multiples of 64 elements
                o.append(torch.nn.functional.pad(part, (0, -part.numel() % 64)))
        return tuple(torch.cat(o) for o in outs)
    nx, ny = c["nx"], c["ny"]
    ec, en, fx, fy = (_at(a, c) for a in _materials(c, seed))
    op = _Op2(c, ec, en)
    pitch = _pitch(nx)
    bx, by = fx, fy
    if c.get("pressure") or kind == "residual":
        p = _at(_pressure(c, seed), c)
        gx, gy = -_diff(p, 1) / op.hx, -_diff(p, 0) / op.hy
        bx, by = fx.clone(), fy.clone()
        bx[:, 1:-1] -= gx
        by[1:-1] -= gy
    if kind == "step":
        vx, vy = torch.zeros_like(fx), torch.zeros_like(fy)
    else:
        vx, vy = (_at(a, c) for a in _velocity(c, seed))
    if kind == "residual":
        s = op.shear(vx, vy)
        ox, oy = torch.zeros_like(vx), torch.zeros_like(vy)
        ox[:, 1:-1] = op.mx(vx, s) + gx
        oy[1:-1] = op.my(vy, s) + gy
        return _padded(pitch, ny, ox), _padded(pitch, ny, oy), _energy(op, bx, by, fx, fy, vx, vy)
    if c.get("variant") == "rbgs":
        _rbgs(op, bx, by, vx, vy, c["sweeps"])
    elif c.get("variant", "ras") == "ras" and c["overlap"] < c["k"] - 1:
        _ras2(c, op, bx, by, vx, vy)
    else:
        _jacobi(op, bx, by, vx, vy, c["sweeps"])
    out = _padded(pitch, ny, vx), _padded(pitch, ny, vy)
    if kind == "step":
        # the energy norm of the result the call has: FP32 leaves its own rounding in the residual
        return out[0], out[1], _energy(op, bx, by, fx, fy, vx, vy) if c["dtype"] == "f64" else None
    return out
