"""The work that a user has this library do: time steps and residuals of the
sub-grid DG shallow-water operator through ``swdg.Context`` / ``swdg.Ensemble``,
the allocation-free residual, and the recorded step with its adjoint.

A case names the call, the terrain and the options; its inputs come from a seed
(rasters and states are made on the GPU) and stand for what ``workloads.py``
describes: the tidal beach, the lagoon on a 2:1 forest, the closed basin and the
paraboloid of the point-sampled mode.  ``exact`` restates the operator and the
step with dense float64 tensor expressions, without the library.
"""
from __future__ import annotations

import math
from types import SimpleNamespace

import numpy as np
import torch

from paper_2505_18743_gb300 import swdg

G = 9.81
PERIOD = 44712.0
# time-step bounds: CFL number per degree (the workloads' own)
CFL = {1: 0.2, 2: 0.12, 3: 0.08}


def _case(name, call, terrain, degree, nx, ny, pix, *, f64_raster=False, mode=0, bulk=False,
          tableau=0, friction=True, members=1, sizes="", host=False, steps=1):
    return dict(name=name, call=call, terrain=terrain, degree=degree, nx=nx, ny=ny, pix=pix,
                f64_raster=f64_raster, mode=mode, bulk=bulk, tableau=tableau, friction=friction,
                members=members, sizes=sizes, host=host, steps=steps)


def listed():
    return [
        # the smallest run: the 16 x 16 degree-1 closed basin, one explicit step; launches count
        _case("basin_step", "step", "basin", 1, 16, 16, 8, f64_raster=True, tableau=1,
              friction=False),
        # a small coastal model coupled through host buffers: state up, 4 steps, state down
        _case("shore_host_steps", "step", "beach", 2, 64, 48, 16, host=True, steps=4),
        # an odd mesh with 5 x 5 pixels per cell, the explicit four-stage scheme, no friction
        _case("odd_rk44_step", "step", "beach", 3, 61, 37, 5, f64_raster=True, tableau=2,
              friction=False),
        # point-sampled bathymetry (the paper's own sampling), a bowl with a moving shoreline
        _case("bowl_points_step", "step", "bowl", 1, 100, 100, 4, f64_raster=True, mode=1),
        # the operator alone inside a pool that forbids allocations
        _case("noalloc_residual", "noalloc", "beach", 2, 96, 64, 16),
        # the operator alone on the 256 x 256 degree-3 tidal beach
        _case("beach_residual", "residual", "beach", 3, 256, 256, 16),
        # the headline: one time step of the 256 x 256 degree-3 tidal beach, FP64
        _case("beach_step", "step", "beach", 3, 256, 256, 16),
        # the same in the FP32-bulk precision
        _case("beach_bulk_step", "step", "beach", 3, 256, 256, 16, bulk=True),
        # non-conforming lagoon: hanging faces, 32/16/8 pixels per cell side, shallow flats
        _case("lagoon_residual", "residual", "lagoon", 2, 128, 64, 32),
        _case("lagoon_step", "step", "lagoon", 2, 128, 64, 32),
        # a parameter sweep: uneven members in one set of launches, FP32-bulk
        _case("sweep_bulk_step", "ensemble", "beach", 2, 0, 0, 8, bulk=True, members=24,
              sizes="32,64,128"),
        # training: one recorded step and its pull-back, the 128 x 128 degree-2 gauge case
        _case("adjoint_step", "adjoint", "beach", 2, 128, 128, 16, f64_raster=True),
    ]


def draw(rng):
    call = rng.choice(["step", "step", "step", "step", "residual", "residual", "ensemble",
                       "adjoint", "noalloc"])
    degree = rng.choice([1, 2, 3, 3])
    bulk = call in ("step", "residual", "ensemble") and rng.random() < 0.3
    terrain = rng.choice(["beach", "beach", "lagoon", "basin", "bowl"])
    cells = math.exp(rng.uniform(math.log(64), math.log(40000)))
    nx = max(4, round(math.sqrt(cells) * math.exp(rng.uniform(-0.4, 0.4))))
    ny = max(4, round(cells / nx))
    pix = rng.choice([3, 4, 5, 8, 11, 16, 32])
    mode = 1 if terrain == "bowl" else 0
    members, sizes = 1, ""
    if call == "ensemble":
        terrain, mode, members = "beach", 0, rng.randrange(2, 25)
        pix = rng.choice([4, 8, 16])
        sizes = ",".join(str(rng.randrange(6, 80)) for _ in range(3))
        nx = ny = 0
    if call == "noalloc":
        terrain, mode = rng.choice(["beach", "basin"]), 0
    if terrain == "lagoon":  # pixels of a coarse cell; about three leaves per coarse cell
        pix = rng.choice([16, 32])
        nx, ny = max(6, nx // 2), max(6, ny // 2)
    if call == "adjoint":
        nx, ny = min(nx, 128), min(ny, 128)
    return {k: v for k, v in _case(
        "", call, terrain, degree, nx, ny, pix, f64_raster=call == "adjoint" or rng.random() < 0.3,
        mode=mode, bulk=bulk, tableau=0 if call == "adjoint" else rng.choice([0, 0, 0, 1, 2, 3]),
        friction=rng.random() < 0.8, members=members, sizes=sizes,
        host=call == "step" and rng.random() < 0.2,
        steps=rng.choice([1, 1, 2]) if call == "step" else 1).items() if k != "name"}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _lobatto(n):
    """n Gauss-Lobatto nodes and weights on [0, 1]"""
    P = np.polynomial.legendre.Legendre.basis(n - 1)
    x = np.concatenate([[-1.0], np.sort(P.deriv().roots().real), [1.0]])
    for _ in range(3):  # polish the interior roots
        x[1:-1] -= P.deriv()(x[1:-1]) / P.deriv(2)(x[1:-1])
    return 0.5 * (1.0 + x), 1.0 / (n * (n - 1) * P(x) ** 2)


def _legendre(n):
    x, w = np.polynomial.legendre.leggauss(n)
    return 0.5 * (1.0 + x), 0.5 * w


def _device():
    return torch.device("cuda" if torch.cuda.is_available() else "cpu")


def _noise(gen, ny, nx, rms):
    """white noise filtered to amplitude 1/|k|, rescaled to rms"""
    dev = _device()
    W = torch.fft.rfft2(torch.randn((ny, nx), generator=gen, device=dev, dtype=torch.float64))
    ky = torch.fft.fftfreq(ny, device=dev, dtype=torch.float64)[:, None]
    kx = torch.fft.rfftfreq(nx, device=dev, dtype=torch.float64)[None, :]
    k = torch.sqrt(kx * kx + ky * ky)
    f = torch.fft.irfft2(W * torch.where(k > 0, 1.0 / k.clamp(min=1e-300), 0.0 * k), s=(ny, nx))
    return f * (rms / f.square().mean().sqrt().clamp(min=1e-300))


def _smooth(rng, X, Y, L, modes=8):
    """low-wavenumber Fourier modes, min-max scaled to [0, 1]"""
    f = torch.zeros_like(X)
    for _ in range(modes):
        kx, ky = rng.integers(0, 4, size=2)
        f += float(rng.standard_normal()) * torch.cos(
            (2 * math.pi / L) * (int(kx) * X + int(ky) * Y) + float(rng.uniform(0, 2 * math.pi)))
    lo, hi = f.min(), f.max()
    return (f - lo) / (hi - lo).clamp(min=1e-300)


def _uniform(nx, ny, Lx, Ly, tag_w):
    hx, hy = Lx / nx, Ly / ny
    i, j = (a.ravel() for a in np.meshgrid(np.arange(nx), np.arange(ny)))
    k = i + nx * j
    nbr = np.full((nx * ny, 4, 2), -1, dtype=np.int32)
    nbr[:, 0, 0] = np.where(i > 0, k - 1, -1 - tag_w)
    nbr[:, 1, 0] = np.where(i < nx - 1, k + 1, -1)
    nbr[:, 2, 0] = np.where(j > 0, k - nx, -1)
    nbr[:, 3, 0] = np.where(j < ny - 1, k + nx, -1)
    return (np.stack([i * hx, j * hy], 1), np.tile([[hx, hy]], (nx * ny, 1)), nbr)


def _forest(level, Lx, Ly, tag_s):
    """leaves of coarse cells refined to level[j, i] in 0..2 (2:1 across coarse cells)"""
    ny0, nx0 = level.shape
    M = 4  # fine cells per coarse side
    own = np.zeros((ny0 * M, nx0 * M), dtype=np.int64)
    lev, gi, gj = [], [], []
    n = 0
    for L in (2, 1, 0):
        J, I = np.nonzero(level == L)
        s = M >> L  # fine cells per leaf side
        for b in range(1 << L):
            for a in range(1 << L):
                ids = n + np.arange(len(I))
                for y in range(s):
                    for x in range(s):
                        own[J * M + b * s + y, I * M + a * s + x] = ids
                lev.append(np.full(len(I), L))
                gi.append(I * M + a * s)
                gj.append(J * M + b * s)
                n += len(I)
    lev, gi, gj = (np.concatenate(v) for v in (lev, gi, gj))
    order = np.lexsort((gi, gj, gi // M, gj // M))
    new = np.empty(n, dtype=np.int64)
    new[order] = np.arange(n)
    own, lev, gi, gj = new[own], lev[order], gi[order], gj[order]
    s = M >> lev
    fx, fy = Lx / (nx0 * M), Ly / (ny0 * M)
    nbr = np.full((n, 4, 2), -1, dtype=np.int32)
    for f in range(4):
        # fine cells just outside the face, at its lower and upper half
        x0 = np.where(f == 0, gi - 1, np.where(f == 1, gi + s, gi))
        y0 = np.where(f == 2, gj - 1, np.where(f == 3, gj + s, gj))
        inside = (x0 >= 0) & (x0 < nx0 * M) & (y0 >= 0) & (y0 < ny0 * M)
        xc, yc = np.clip(x0, 0, nx0 * M - 1), np.clip(y0, 0, ny0 * M - 1)
        a = own[yc, xc]
        up = s // 2
        b = own[np.clip(yc + (up if f < 2 else 0), 0, ny0 * M - 1),
                np.clip(xc + (up if f >= 2 else 0), 0, nx0 * M - 1)]
        nbr[:, f, 0] = np.where(inside, a, -1 - (tag_s if f == 2 else 0))
        nbr[:, f, 1] = np.where(inside & (lev[a] > lev), b, -1)
    return (np.stack([gi * fx, gj * fy], 1), np.stack([s * fx, s * fy], 1), nbr)


def _raster(case, nx, ny, gen, rng):
    """depth [ny pix, nx pix] (positive down) on the device, and the domain size"""
    dev, pix, kind = _device(), case["pix"], case["terrain"]
    my, mx = ny * pix, nx * pix
    u = ((torch.arange(mx, device=dev, dtype=torch.float64) + 0.5) / mx)[None, :]
    v = ((torch.arange(my, device=dev, dtype=torch.float64) + 0.5) / my)[:, None]
    if kind == "beach":  # 30 m deep, a beach over the last quarter, noise and channels
        Lx, Ly = 20000.0, 20000.0 * ny / nx
        z = torch.where(u < 0.75, 30.0 + 0 * u, 30.0 - 140.0 * (u - 0.75)) + _noise(gen, my, mx, 1.5)
        for _ in range(8):
            walk = torch.cumsum(torch.randn(mx, generator=gen, device=dev, dtype=torch.float64), 0)
            yc = (float(rng.uniform(0.1, 0.9)) * my + walk).clamp(0, my - 1)[None, :]
            half = 0.5 * int(rng.integers(3, 6))
            z += 3.0 * ((u >= 0.75) & ((v * my - yc).abs() < half))
    elif kind == "lagoon":  # open sea, a barrier with two inlets, a shallow lagoon with flats
        Lx, Ly = 50000.0, 50000.0 * ny / nx
        x, y = u * Lx, v * Ly
        coast = _coast(u) * Ly
        d = y - coast
        flats = _noise(gen, my, mx, 1.0)
        lag = 1.75 + 1.25 * torch.sin(x / 2300.0 + 1.3) * torch.cos(y / 1700.0)
        lag = torch.where(flats > 0.9, 0.3 * torch.tanh(flats - 1.2), lag)
        sea = 3.0 + 12.0 * (-d / 8000.0).clamp(0, 1)
        z = torch.where(d < -300.0, sea, torch.where(d > 300.0, lag, -2.0 + 0 * lag))
        for xi in (0.3 * Lx, 0.68 * Lx):
            cut = ((x - xi).abs() < 250.0) & (d.abs() < 900.0)
            z = torch.where(cut, 15.0 - d.abs() / 90.0, z)
    elif kind == "basin":  # 10 m deep, a bump and random steps
        Lx, Ly = 1000.0, 1000.0 * ny / nx
        x, y = u * Lx, v * Ly
        z = 10.0 - 6.0 * torch.exp(-((x - 0.5 * Lx) ** 2 + (y - 0.5 * Ly) ** 2) / 150.0 ** 2)
        for _ in range(20):
            a, b, w, h = rng.uniform(0, 1, 2).tolist() + rng.uniform(0.05, 0.3, 2).tolist()
            z = z + float(rng.choice([-2.0, 2.0])) * ((u >= a) & (u < a + w) & (v >= b) & (v < b + h))
    else:  # a paraboloid bowl
        Lx, Ly = 3.0, 3.0 * ny / nx
        z = 0.1 * (1.0 - ((u * Lx - 0.5 * Lx) ** 2 + (v * Ly - 0.5 * Ly) ** 2))
    return (z if case["f64_raster"] else z.float()), Lx, Ly


def _coast(u):
    """the lagoon's coastline as a fraction of the domain height, at abscissae u
    in [0, 1]: one shore, so that the mesh refined toward it is the same for
    every seed"""
    f = torch.full_like(u, 0.4)
    for m, (a, p) in enumerate(((0.06, 0.3), (-0.04, 2.1), (0.03, 4.4), (0.02, 1.2), (-0.016, 5.0)), 1):
        f = f + a * torch.sin(2 * math.pi * m * u + p)
    return f


def _levels(nx, ny):
    """refinement level of every coarse cell of the lagoon, 2:1 across them"""
    u = (torch.arange(nx, dtype=torch.float64)[None, :] + 0.5) / nx
    d = np.abs((np.arange(ny)[:, None] + 0.5) / ny - _coast(u).numpy())
    level = (d < 0.25).astype(int) + (d < 0.12)
    for _ in range(2):
        p = np.pad(level, 1)
        level = np.maximum(level, np.max([p[1:-1, :-2], p[1:-1, 2:], p[:-2, 1:-1], p[2:, 1:-1]],
                                         axis=0) - 1)
    return level


def _domain(case, nx, ny, seed):
    """mesh, raster and state of one (member) domain, from the seed alone"""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device=_device())
    gen.manual_seed(int(seed))
    z, Lx, Ly = _raster(case, nx, ny, gen, rng)
    kind = case["terrain"]
    if kind == "lagoon":
        x0y0, hxhy, nbr = _forest(_levels(nx, ny), Lx, Ly, 1)
    else:
        x0y0, hxhy, nbr = _uniform(nx, ny, Lx, Ly, 1 if kind == "beach" else 0)
    s, _ = _lobatto(case["degree"] + 1)
    m = case["degree"] + 1
    dev = _device()
    x0, h = torch.tensor(x0y0, device=dev), torch.tensor(hxhy, device=dev)
    X = x0[:, :1] + h[:, :1] * torch.tensor(np.tile(s, m), device=dev)
    Y = x0[:, 1:] + h[:, 1:] * torch.tensor(np.repeat(s, m), device=dev)
    c = _smooth(rng, X, Y, Lx)
    wave, sx, sy = (_smooth(rng, X, Y, Lx) for _ in range(3))
    if kind == "bowl":  # a tilted surface and a slow stream over the wet part
        zeta = 0.02 * (wave - 0.5) + 0.01 * (X / Lx - 0.5)
        depth = 0.1 * (1.0 - ((X - 0.5 * Lx) ** 2 + (Y - 0.5 * Ly) ** 2)) + zeta
        wet, speed = depth.clamp(min=0.0), 0.2
    else:
        zeta = (0.1 if kind == "basin" else 0.4) * wave
        # depth of the shallowest point of each cell bounds its discharge
        P = torch.tensor(np.rint(hxhy[:, 0] / (Lx / z.shape[1])).astype(np.int64), device=dev)
        lo = torch.empty(len(x0y0), device=dev, dtype=torch.float64)
        for p in torch.unique(P).tolist():
            sel = P == p
            blocks = -torch.nn.functional.max_pool2d(-z[None, None].double(), p)[0, 0]
            ij = torch.round(x0[sel] / h[sel]).long()
            lo[sel] = blocks[ij[:, 1], ij[:, 0]]
        wet, speed = lo.clamp(0.0, 3.0)[:, None], 0.3
    qx, qy = speed * wet * (sx - 0.4), speed * wet * (sy - 0.5)
    n = len(x0y0)
    man = np.full(n, 0.02 if case["friction"] else 0.0)
    if case["friction"]:
        man *= 0.7 + 0.6 * rng.random(n)
    return SimpleNamespace(n=n, x0y0=x0y0, hxhy=hxhy, nbr=nbr, z=z, dx=Lx / z.shape[1],
                           dy=Ly / z.shape[0], u=[a.contiguous() for a in (zeta, qx, qy, c)],
                           man=man, amp=1.0)


def _domains(case, seed):
    if case["members"] == 1:
        return [_domain(case, case["nx"], case["ny"], seed)]
    sizes = [int(v) for v in case["sizes"].split(",")]
    out = []
    for m in range(case["members"]):
        N = sizes[(5 * m + m // 3) % len(sizes)]
        d = _domain(case, N, N, seed * 1000 + m)
        d.amp = 0.2 + 1.3 * m / case["members"]
        out.append(d)
    return out


def _field_config(case):
    field = case["terrain"] in ("beach", "lagoon")  # metres of water over kilometres
    eps = 0.1 if field else 0.01 if case["terrain"] == "basin" else 1e-3
    return dict(degree=case["degree"], subgrid_mode=case["mode"], tableau=case["tableau"], g=G,
                eps_vel=eps, h_lim=eps, eps0=1e-6, cfl=CFL[case["degree"]])


T0 = 3000.0  # the tide stands about 0.4 m up


def prepare(case, seed):
    doms = _domains(case, seed)
    cfg = _field_config(case)
    s = SimpleNamespace(case=case, t=T0)
    if case["call"] == "noalloc":
        d = doms[0]
        dev = _device()
        s.cfg = swdg.swdg_config(cfg["degree"], 0, 0, 0, G, cfg["eps_vel"], cfg["h_lim"],
                                 cfg["eps0"], cfg["cfl"], 20, 1e-12, None)
        P = case["pix"]
        ny, nx = d.z.shape[0] // P, d.z.shape[1] // P
        s.args = (d.n, torch.tensor(d.hxhy, device=dev), torch.tensor(d.nbr, device=dev),
                  d.z.reshape(ny, P, nx, P).permute(0, 2, 1, 3).contiguous(), P,
                  swdg.SWDG_PIX_F64 if case["f64_raster"] else swdg.SWDG_PIX_F32,
                  torch.tensor(d.man, device=dev), torch.stack(d.u).contiguous(), T0)
        s.out = torch.empty((6, d.n, (cfg["degree"] + 1) ** 2), device=dev, dtype=torch.float64)
        s.dt = torch.empty(1, device=dev, dtype=torch.float64)
        s.bc = [(1, swdg.SWDG_BC_TIDE, 1.0, PERIOD, 0.0)]
        return s
    cls = swdg.Ensemble if case["call"] == "ensemble" else swdg.Context
    ctx = cls(precision=1 if case["bulk"] else 0, **cfg)
    if case["call"] == "ensemble":
        first = np.concatenate([[0], np.cumsum([d.n for d in doms])])
        nbr = np.concatenate([np.where(d.nbr >= 0, d.nbr + f, d.nbr)
                              for d, f in zip(doms, first)]).astype(np.int32)
        ctx.upload_mesh(np.concatenate([d.x0y0 for d in doms]),
                        np.concatenate([d.hxhy for d in doms]), nbr)
        ctx.set_members(first)
        ctx.upload_bathymetry_members([SimpleNamespace(z=d.z.cpu().numpy(), xo=0.0, yo=0.0, dx=d.dx,
                                                       dy=d.dy) for d in doms])
        for m, d in enumerate(doms):
            ctx.set_boundary_member(m, 1, swdg.SWDG_BC_TIDE, d.amp, PERIOD, 0.0)
    else:
        d = doms[0]
        ctx.upload_mesh(d.x0y0, d.hxhy, d.nbr)
        ctx.upload_bathymetry(d.z.cpu().numpy(), 0.0, 0.0, d.dx, d.dy)
        ctx.set_boundary(1, swdg.SWDG_BC_TIDE, 1.0, PERIOD, 0.0)
    ctx.set_manning(np.concatenate([d.man for d in doms]))
    s.ctx = ctx
    s.u = [torch.cat([d.u[f] for d in doms]).contiguous() for f in range(4)]
    if case["host"]:
        s.u = [a.cpu().numpy() for a in s.u]
        s.out = None
    else:
        s.out = [torch.empty_like(s.u[0]) for _ in range(6 if case["call"] == "residual" else 4)]
    if case["call"] == "residual":
        ctx.set_state(*s.u)
    if case["call"] == "adjoint":
        gen = torch.Generator(device=_device())
        gen.manual_seed(int(seed) + 7)
        s.cot = [torch.randn(a.shape, generator=gen, device=a.device, dtype=torch.float64)
                 for a in s.u]
        # half of the positivity bound of the fastest point: a fixed step, as in a re-run block
        h = float(doms[0].hxhy.min())
        s.dt = 0.5 * cfg["cfl"] * h / (2.0 + math.sqrt(G * 40.0))
    return s


def run(s):
    call = s.case["call"]
    if call == "noalloc":
        swdg.residual_noalloc(s.cfg, *s.args, s.out, s.dt, s.bc)
        return s.out, s.dt
    ctx = s.ctx
    if call == "residual":
        return ctx.residual(s.t, s.out)
    ctx.set_state(*s.u)
    if call == "adjoint":
        ctx.step_record(s.dt, s.t)
        return ctx.get_state(s.out), ctx.step_vjp(s.cot)
    if call == "ensemble":
        ctx.set_times(s.t)
        ctx.step(s.case["steps"])
        return ctx.get_state(s.out)
    t = ctx.step(s.case["steps"], t=s.t)
    return ctx.get_state(s.out), t


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _cells(case):
    if case["members"] > 1:
        sizes = [int(v) for v in case["sizes"].split(",")]
        return sum(sizes[(5 * m + m // 3) % len(sizes)] ** 2 for m in range(case["members"]))
    if case["terrain"] == "lagoon":
        return int((4 ** _levels(case["nx"], case["ny"])).sum())
    return case["nx"] * case["ny"]


def work(case):
    """Bytes: the state, the residual, the pixels and the geometry once per
    operator evaluation and the state, mass and residual fields once per stage
    solve.  Flops: the sum-factorised contractions (multiply and add), about 70
    per volume and 110 per face point, and the stage solves (two contraction
    pairs for the continuity, four for the momentum, a Cholesky solve and two
    refinement passes for the tracer)."""
    r = case["degree"]
    n1, nv, nm = r + 1, (3 * r) // 2 + 1, r + 2
    nd = n1 * n1
    n = _cells(case)
    pixel = case["pix"] ** 2 * (8 if case["f64_raster"] else 4)
    if case["terrain"] == "lagoon":
        pixel *= case["nx"] * case["ny"] / n  # the leaves of a coarse cell share its pixels
    if case["mode"] == 1:
        pixel = 8 * (nv * nv + nm * nm + n1 * n1)
    geom = 8 * 5 + 32
    res_b = 8 * 10 * nd + pixel + geom
    xy = lambda m: n1 * m * (n1 + m)  # noqa: E731  one 2D contraction, multiply-adds
    res_f = 2 * (6 * xy(nv) + 9 * xy(nv)) + 70 * nv * nv + 2 * nm * (2 * 8 * n1 + 110) + 32 * nm * n1
    st_b = 8 * (4 + 2 + 6 + 4) * nd + pixel
    st_f = 2 * (2 * xy(nm) + 2 * nd * n1 + 6 * xy(n1) + 4 * xy(nm) + nd ** 3 // 6) + 20 * nm * nm
    s = {0: 3, 1: 3, 2: 4, 3: 1}[case["tableau"]]
    step_b, step_f = s * (res_b + st_b) + 8 * 6 * nd, s * (res_f + st_f) + 4 * xy(nm) + 10 * nm * nm
    k = case["steps"]
    if case["call"] in ("residual", "noalloc"):
        b, f = res_b, res_f
    elif case["call"] == "adjoint":  # the step, and about three times its work pulling it back
        b, f = 3 * step_b, 4 * step_f
    else:
        b, f = k * step_b, k * step_f
    return {"bytes": float(n * b), "flops": float(n * f)}


# ---------------------------------------------------------------------------
# the operator and the step in dense float64 expressions
# ---------------------------------------------------------------------------
def _lagrange(xs, x):
    """values and derivatives [len(x), len(xs)] of the nodal basis"""
    v, d = np.ones((len(x), len(xs))), np.zeros((len(x), len(xs)))
    for a in range(len(xs)):
        others = [b for b in range(len(xs)) if b != a]
        for b in others:
            v[:, a] *= (x - xs[b]) / (xs[a] - xs[b])
        for k in others:
            t = np.full(len(x), 1.0 / (xs[a] - xs[k]))
            for b in others:
                if b != k:
                    t *= (x - xs[b]) / (xs[a] - xs[b])
            d[:, a] += t
    return v, d


def _overlap(edges, P):
    """[len(edges) - 1, P]: share of each sub-interval that each of P pixels covers"""
    lo, hi = np.array(edges[:-1])[:, None] * P, np.array(edges[1:])[:, None] * P
    p = np.arange(P)[None, :]
    return np.maximum(0.0, np.minimum(hi, p + 1) - np.maximum(lo, p)) / (hi - lo)


def _edges(w):
    e = np.concatenate([[0.0], np.cumsum(w)])
    e[-1] = 1.0
    return e


TABLEAUX = {
    1: ([[0, 0, 0], [1, 0, 0], [.25, .25, 0]], [1 / 6, 1 / 6, 2 / 3], [0, 1, .5]),
    2: ([[0] * 4, [.5, 0, 0, 0], [0, .5, 0, 0], [0, 0, 1, 0]], [1 / 6, 1 / 3, 1 / 3, 1 / 6],
        [0, .5, .5, 1]),
    3: ([[0]], [1], [0]),
}


def _tableau(which):
    if which:
        a, b, c = TABLEAUX[which]
        return a, a, b, b, c
    g = 2 - math.sqrt(2)  # TR-BDF2 and its explicit companion
    d, w = 1 - 1 / math.sqrt(2), 1 / (2 * math.sqrt(2))
    return ([[0, 0, 0], [g, 0, 0], [.5, .5, 0]], [[0, 0, 0], [d, d, 0], [w, w, d]], [w, w, d],
            [w, w, d], [0, g, 1])


class _Exact:
    def __init__(self, case, doms):
        self.cfg = _field_config(case)
        self.mode = case["mode"]
        r = case["degree"]
        first = np.concatenate([[0], np.cumsum([d.n for d in doms])])
        self.n = n = int(first[-1])
        t = lambda a: torch.tensor(np.asarray(a), dtype=torch.float64)  # noqa: E731
        self.memb = torch.tensor(np.repeat(np.arange(len(doms)), [d.n for d in doms]))
        self.amp = t([d.amp for d in doms])
        h = np.concatenate([d.hxhy for d in doms])
        self.hx, self.hy = t(h[:, :1]), t(h[:, 1:])
        self.J = self.hx * self.hy
        self.man = t(np.concatenate([d.man for d in doms]))
        nbr = np.concatenate([np.where(d.nbr >= 0, d.nbr + f, d.nbr) for d, f in zip(doms, first)])
        xs, _ = _lobatto(r + 1)
        self.n1 = r + 1
        xv, wv = _legendre((3 * r) // 2 + 1)
        xm, wm = _lobatto(r + 2)
        xg, wg = _legendre(r + 1)
        self.nm = r + 2
        kron = lambda y, x: t(np.kron(y, x))  # noqa: E731  point index x fastest
        (bv, dv), (bm, _), (bg, _) = (_lagrange(xs, x) for x in (xv, xm, xg))
        self.Bv, self.Dx, self.Dy, self.wv = kron(bv, bv), kron(bv, dv), kron(dv, bv), t(np.kron(wv, wv))
        self.Bm, self.wm2 = kron(bm, bm), t(np.kron(wm, wm))
        self.Bg, self.wg2 = kron(bg, bg), t(np.kron(wg, wg))
        # 1D traces along a face: 0 whole, 1 / 2 its lower / upper half
        halves = [(xm, _edges(wm))] + [(0.5 * (xm + k), 0.5 * (_edges(wm) + k))
                                       for k in (0, 1)]
        self.tr = [t(_lagrange(xs, x)[0]) for x, _ in halves]
        self.wm = t(wm)
        # 1D sampling: cell sets v, m, g and the face strips m0, m1 (normal), h0, h1, h2 (along)
        em = _edges(wm)
        self.sets = {"v": (_edges(wv), xv), "m": (em, xm), "g": (_edges(wg), xg),
                     "m0": (em[:2], xm[:1]), "m1": (em[-2:], xm[-1:])}
        self.sets.update({"h%d" % k: (e, x) for k, (x, e) in enumerate(halves)})
        self.cls = []  # (cells, tiles [m, P, P]) per pixel count
        if self.mode == 0:
            for d, f in zip(doms, first):
                P = np.rint(d.hxhy[:, 0] / d.dx).astype(int)
                z = d.z.cpu().double().numpy()
                for p in np.unique(P):
                    k = np.nonzero(P == p)[0]
                    ij = np.rint(d.x0y0[k] / d.hxhy[k]).astype(int)
                    bl = z.reshape(z.shape[0] // p, p, z.shape[1] // p, p).transpose(0, 2, 1, 3)
                    self.cls.append((torch.tensor(k + f), t(bl[ij[:, 1], ij[:, 0]])))
            byp = {}
            for k, tl in self.cls:
                byp.setdefault(tl.shape[1], []).append((k, tl))
            self.cls = [(torch.cat([a for a, _ in v]), torch.cat([b for _, b in v]))
                        for v in byp.values()]
            self.cid, self.row = torch.empty(n, dtype=torch.long), torch.empty(n, dtype=torch.long)
            self.zmin, self.zmax = torch.empty(n, dtype=torch.float64), torch.empty(n, dtype=torch.float64)
            for q, (k, tl) in enumerate(self.cls):
                self.cid[k], self.row[k] = q, torch.arange(len(k))
                self.zmin[k], self.zmax[k] = tl.amin((1, 2)), tl.amax((1, 2))
        else:
            d = doms[0]
            self.dom, self.zr = d, d.z.cpu().double().numpy()
            zz = self.samples(torch.arange(n), "m", "m")
            self.zmax = zz.amax(1)
        self.zc = {}
        # faces: groups of equal direction and kinds (own trace, neighbour trace)
        self.groups = []
        lev = torch.tensor(h[:, 0])
        for f in range(4):
            s0, s1 = torch.tensor(nbr[:, f, 0]).long(), torch.tensor(nbr[:, f, 1]).long()
            k = torch.arange(n)
            b = s0 < 0
            for tag in torch.unique(s0[b]).tolist():
                self.groups.append((f, k[s0 == tag], None, 0, 0, -1 - tag))
            for half, s in ((1, s0), (2, s1)):
                sel = s1 >= 0
                if bool(sel.any()):
                    self.groups.append((f, k[sel], s[sel], half, 0, None))
            c = ~b & (s1 < 0)
            nb = s0.clamp(min=0)
            same = c & (lev[nb] < 1.5 * lev)
            if bool(same.any()):
                self.groups.append((f, k[same], s0[same], 0, 0, None))
            fine = c & ~same  # which half of the coarse neighbour's face this cell is
            up = torch.tensor(nbr)[nb, f ^ 1, 1].long() == k
            for half in (1, 2):
                sel = fine & (up == (half == 2))
                if bool(sel.any()):
                    self.groups.append((f, k[sel], s0[sel], 0, half, None))

    def samples(self, k, sx, sy):
        """mode P: bilinear depth at the tensor points of the sets sx, sy of cells k"""
        d, z = self.dom, self.zr
        X = d.x0y0[k.numpy(), 0][:, None] + self.hx[k].numpy() * self.sets[sx][1][None, :]
        Y = d.x0y0[k.numpy(), 1][:, None] + self.hy[k].numpy() * self.sets[sy][1][None, :]
        fi = np.clip(X / d.dx - 0.5, 0, z.shape[1] - 1)[:, None, :]
        fj = np.clip(Y / d.dy - 0.5, 0, z.shape[0] - 1)[:, :, None]
        i = np.minimum(np.floor(fi).astype(int), z.shape[1] - 2)
        j = np.minimum(np.floor(fj).astype(int), z.shape[0] - 2)
        a, b = fi - i, fj - j
        out = (1 - a) * (1 - b) * z[j, i] + a * (1 - b) * z[j, i + 1] + \
            (1 - a) * b * z[j + 1, i] + a * b * z[j + 1, i + 1]
        return torch.tensor(out.reshape(len(k), X.shape[1] * Y.shape[1]))

    def VA(self, k, eta, sx, sy):
        """sub-grid depth and wet area at the points of the sets sx, sy of cells k"""
        key = (sx, sy)
        if self.mode == 1:
            e = eta + self.samples(k, sx, sy)
            return e.clamp(min=0.0), (e > 0).double()
        if key not in self.zc:  # mean depth of every sub-cell
            zb = torch.empty((self.n, eta.shape[1]), dtype=torch.float64)
            for kk, tl in self.cls:
                P = tl.shape[1]
                wx, wy = (torch.tensor(_overlap(self.sets[s][0], P)) for s in (sx, sy))
                zb[kk] = torch.einsum("bj,ai,kji->kba", wy, wx, tl).reshape(len(kk), -1)
            self.zc[key] = zb
        V, A = eta + self.zc[key][k], torch.ones_like(eta)
        hi, lo = eta.amax(1), eta.amin(1)
        dry = hi <= -self.zmax[k]
        V[dry], A[dry] = 0.0, 0.0
        mixed = ~dry & ~(lo > -self.zmin[k])
        for q, (_, tl) in enumerate(self.cls):
            sel = torch.nonzero(mixed & (self.cid[k] == q)).flatten()
            if not len(sel):
                continue
            tls, P = tl[self.row[k[sel]]], tl.shape[1]
            wx, wy = (_overlap(self.sets[s][0], P) for s in (sx, sy))
            for p in range(eta.shape[1]):
                ax, by = wx[p % len(wx)], wy[p // len(wx)]
                ix, jy = np.nonzero(ax)[0], np.nonzero(by)[0]
                w = torch.tensor(np.outer(by[jy], ax[ix]))
                d = eta[sel, p][:, None, None] + tls[:, jy[0]:jy[-1] + 1, ix[0]:ix[-1] + 1]
                V[sel, p] = (w * d.clamp(min=0.0)).sum((1, 2))
                A[sel, p] = (w * (d > 0)).sum((1, 2))
        return V, A

    def vel(self, h):
        e, hs = self.cfg["eps_vel"], torch.where(h > 0, h, torch.ones_like(h))
        f = torch.where(hs >= e, 1.0 / hs, math.sqrt(2.0) * hs / torch.sqrt(e ** 4 + hs ** 4))
        return torch.where(h > 0, f, torch.zeros_like(h))

    def gamma(self, n, h, qx, qy):
        f = self.vel(h)  # 1 / h_des
        return G * n * n * torch.sqrt(qx * qx + qy * qy) * f ** (7.0 / 3.0)

    def residual(self, u, t, dt=False):
        """the six residual fields; with dt also max lambda l / J per member"""
        n, cells = self.n, torch.arange(self.n)
        hx, hy, w = self.hx, self.hy, self.J * self.wv
        z, qx, qy, c = (a @ self.Bv.T for a in u)
        zx, zy = u[0] @ self.Dx.T / hx, u[0] @ self.Dy.T / hy
        h, _ = self.VA(cells, z, "v", "v")
        f = self.vel(h)
        ux, uy = f * qx, f * qy
        gam = self.gamma(self.man[:, None], h, qx, qy)

        def integ(a, b, v=None):
            out = (w * a / hx) @ self.Dx + (w * b / hy) @ self.Dy
            return out if v is None else out + (w * v) @ self.Bv

        out = [integ(qx, qy), integ(qx * ux, qx * uy, -G * h * zx), integ(qy * ux, qy * uy, -G * h * zy),
               integ(c * qx, c * qy), (w * -gam * qx) @ self.Bv, (w * -gam * qy) @ self.Bv]
        rate = torch.zeros(len(self.amp), dtype=torch.float64)
        n1, m = self.n1, self.nm
        node = [[n1 * j for j in range(n1)], [n1 - 1 + n1 * j for j in range(n1)],
                list(range(n1)), [j + n1 * (n1 - 1) for j in range(n1)]]
        for f, k, nb, ho, hn, tag in self.groups:
            sg, ax = (-1.0, 1.0)[f & 1], f >> 1
            nx, ny = (sg, 0.0) if ax == 0 else (0.0, sg)

            def side(cell, face, half):
                nrm = "m%d" % (face & 1)
                s = (nrm, "h%d" % half) if face < 2 else ("h%d" % half, nrm)
                return [a[cell][:, node[face]] @ self.tr[half].T for a in u], \
                    lambda e: self.VA(cell, e, *s)[0]

            (zm, qxm, qym, cm), Vm = side(k, f, ho)
            if nb is not None:
                (zp, qxp, qyp, cp), Vp = side(nb, f ^ 1, hn)
            else:
                zp, qxp, qyp, cp, Vp = zm, qxm, qym, cm, Vm
                if tag == 1:
                    tide = self.amp[self.memb[k]] * torch.sin(2 * math.pi * t[self.memb[k]] / PERIOD)
                    zp = tide[:, None].expand(-1, m).contiguous()
                else:
                    qn = qxm * nx + qym * ny
                    qxp, qyp = qxm - 2 * qn * nx, qym - 2 * qn * ny
            hm, hp = Vm(zm), Vp(zp)
            if nb is not None:
                hsm, hsp = torch.minimum(hm, Vp(zm)), torch.minimum(hp, Vm(zp))
            else:
                hsm, hsp = hm, hp
            fm, fp = self.vel(hm), self.vel(hp)
            umx, umy, upx, upy = fm * qxm, fm * qym, fp * qxp, fp * qyp
            unm, unp = umx * nx + umy * ny, upx * nx + upy * ny
            lam = torch.maximum(unm.abs() + torch.sqrt(G * hm), unp.abs() + torch.sqrt(G * hp))
            a, b, c1, d1 = hsm * umx, hsm * umy, hsp * upx, hsp * upy
            pres = 0.25 * G * (hsm + hsp) * (hsm - hsp)
            flux = [0.5 * ((a + c1) * nx + (b + d1) * ny) + 0.5 * lam * (hsm - hsp),
                    0.5 * (a * unm + c1 * unp) + 0.5 * lam * (a - c1) - pres * nx,
                    0.5 * (b * unm + d1 * unp) + 0.5 * lam * (b - d1) - pres * ny,
                    0.5 * ((a * cm + c1 * cp) * nx + (b * cm + d1 * cp) * ny)
                    + 0.5 * lam * (hsm * cm - hsp * cp)]
            L = (self.hy if ax == 0 else self.hx)[k] * (0.5 if ho else 1.0)
            for q in range(4):
                out[q][k[:, None], torch.tensor(node[f])[None, :]] -= (L * self.wm * flux[q]) @ self.tr[ho]
            if dt:
                v = (lam.clamp(min=1e-12) * L / self.J[k]).amax(1)
                rate.scatter_reduce_(0, self.memb[k], v, "amax")
        return (out, rate) if dt else out

    def H(self, k, zeta):
        V, A = self.VA(k, zeta @ self.Bm.T, "m", "m")
        return V, A

    def hbar(self, k, e):
        w = self.J[k] * self.wm2
        V, A = self.VA(k, e[:, None].expand(-1, len(self.wm2)).contiguous(), "m", "m")
        return (w * V).sum(1), (w * A).sum(1)

    def level(self, k, target, e):
        """constant elevations with wet mass `target` on cells k"""
        _, A = self.hbar(k, e)
        e = torch.where(A == 0, -self.zmax[k] + self.cfg["eps0"], e)
        for _ in range(20):
            Hk, A = self.hbar(k, e)
            e = e - torch.where(A > 0, (Hk - target) / A.clamp(min=1e-300), torch.zeros_like(e))
        return e

    def begin(self, u):
        u = [a.clone() for a in u]
        cells = torch.arange(self.n)
        w, J = self.J * self.wm2, self.J[:, 0]
        V, _ = self.H(cells, u[0])
        flag = V.amin(1) > self.cfg["h_lim"]
        k = torch.nonzero(~flag).flatten()
        if len(k):
            wk, Vk, ck = w[k], V[k], u[3][k] @ self.Bm.T
            mass, tr = (wk * Vk).sum(1), (wk * Vk * ck).sum(1)
            mean = [(self.wg2 * (u[f][k] @ self.Bg.T)).sum(1) for f in (1, 2, 3)]
            wet = mass > 1e-14 * J[k] * self.cfg["h_lim"]
            cn = torch.where(wet, tr / mass.clamp(min=1e-300), mean[2])
            e = -self.zmax[k]
            p = mass > 0
            e[p] = self.level(k[p], mass[p], (u[0][k] @ self.Bm.T).amax(1)[p])
            for f, v in ((0, e), (1, mean[0]), (2, mean[1]), (3, cn)):
                same = (u[f][k] == u[f][k][:, :1]).all(1)
                u[f][k] = torch.where(same[:, None], u[f][k], v[:, None].expand_as(u[f][k]))
            V[k], _ = self.H(k, u[0][k])
        wc = w * V * (u[3] @ self.Bm.T)
        return u, flag, (w * V) @ self.Bm, (w * V).sum(1), wc @ self.Bm, wc.sum(1)

    def mass(self, wgt):
        return torch.einsum("pi,kp,pj->kij", self.Bm, wgt, self.Bm)

    def stage(self, un, prev, res, wa, wat, add, b0, flag, dt, llin):
        HN, HNb, CN, CNb = b0
        cells, J = torch.arange(self.n), self.J[:, 0]
        F = sum(a * r[0] for a, r in zip(wa, res))
        T, Tb = HN + dt[:, None] * F, HNb + dt * F.sum(1)
        rq = [dt[:, None] * sum(a * r[1 + f] + b * r[4 + f] for a, b, r in zip(wa, wat, res))
              for f in (0, 1)]
        rc = CN + dt[:, None] * sum(a * r[3] for a, r in zip(wa, res))
        w = self.J * self.wm2
        z, full = un[0].clone(), flag.clone()
        act = torch.nonzero(full).flatten()
        for _ in range(20):  # Newton on the wet mass
            V, A = self.H(act, z[act])
            dry = (A == 0).any(1)
            full[act[dry]] = False
            act, V, A = act[~dry], V[~dry], A[~dry]
            if not len(act):
                break
            d = torch.linalg.solve(self.mass(w[act] * A), (w[act] * V) @ self.Bm - T[act])
            z[act] -= d
            act = act[~(d.abs().sum(1) <= 1e-13 * (1.0 + z[act].abs()).sum(1))]
        k = torch.nonzero(full).flatten()
        full[k] = ~(self.H(k, z[k])[1] == 0).any(1)
        sc = torch.nonzero(~full).flatten()
        k = torch.nonzero(full).flatten()
        # momentum
        wg = self.J * self.wg2
        gam = torch.zeros_like(wg)
        if add:
            Vg, _ = self.VA(cells, prev[0] @ self.Bg.T, "g", "g")
            gam = self.gamma(self.man[:, None], Vg, prev[1] @ self.Bg.T, prev[2] @ self.Bg.T)
        D = wg * (1.0 + add * dt[:, None] * gam)
        Am = torch.einsum("pi,kp,pj->kij", self.Bg, D, self.Bg)
        q = [torch.linalg.solve(Am, rq[f] + (wg * (un[1 + f] @ self.Bg.T)) @ self.Bg) for f in (0, 1)]
        c = un[3].clone()
        if len(k):
            Vk, _ = self.H(k, z[k])
            c[k] = torch.linalg.solve(self.mass(w[k] * Vk), rc[k])
        if len(sc):
            z0 = un[0][sc]
            e = self.level(sc, Tb[sc], (self.wm2 * (z0 @ self.Bm.T)).sum(1))
            z[sc] = e[:, None].expand_as(z0)
            for f in (0, 1):
                v = ((wg * (un[1 + f] @ self.Bg.T)).sum(1) + rq[f].sum(1)) / D.sum(1)
                q[f][sc] = v[sc][:, None].expand_as(z0)
            Hs, _ = self.hbar(sc, e)
            v = (CNb[sc] + (rc - CN)[sc].sum(1)) / Hs.clamp(min=1e-300)
            c[sc] = torch.where((Hs > 1e-14 * J[sc] * self.cfg["h_lim"])[:, None],
                                v[:, None].expand_as(z0), un[3][sc])
        ll = [-(wg * gam * (q[f] @ self.Bg.T)) @ self.Bg for f in (0, 1)] if llin else None
        return [z, q[0], q[1], c], full, ll

    def step(self, u, t):
        a, at, b, bt, c = _tableau(self.cfg["tableau"])
        s = len(b)
        un, flag, *b0 = self.begin(u)
        stages, res, ll = [un], [], None
        for l in range(s):
            if l:
                v, flag, m = self.stage(un, stages[-1], res, a[l][:l], at[l][:l], at[l][l], b0, flag,
                                        dt, l == s - 1 and at[l][l] != 0)
                ll = m or ll
                stages.append(v)
                res.append(self.residual(v, t + c[l] * dtm))
            else:
                r, rate = self.residual(un, t, dt=True)
                dtm = self.cfg["cfl"] / rate
                dt = dtm[self.memb]
                res.append(r)
        if ll is not None:
            res[-1] = res[-1][:4] + ll
        out, _, _ = self.stage(un, stages[-1], res, b, bt, 0.0, b0, flag, dt, False)
        return out, t + dtm


def exact(case, seed):
    """None for the adjoint: its value is a derivative along the path that the
    forward step's own decisions took."""
    if case["call"] == "adjoint":
        return None
    doms = _domains(case, seed)
    x = _Exact(case, doms)
    u = [torch.cat([d.u[f].cpu() for d in doms]) for f in range(4)]
    t = torch.full((len(doms),), T0, dtype=torch.float64)
    if case["call"] == "noalloc":
        out, rate = x.residual(u, t, dt=True)
        return torch.stack(out), x.cfg["cfl"] / rate
    if case["call"] == "residual":
        return dict(zip(("F", "Gx", "Gy", "R", "Lx", "Ly"), x.residual(u, t)))
    for _ in range(case["steps"]):
        u, t = x.step(u, t)
    return u if case["call"] == "ensemble" else (u, float(t[0]))
