"""The FP32-bulk path gives the same bits as it did when they were recorded.

FP64 values are rounded to FP32 throughout this path, so a sum of another order
or arithmetic in its FP64 parts does not stay at 1e-16: where it moves a value
across an FP32 rounding boundary the result moves by 1.2e-7 of that value.  The
recorded digests (tests/golden/fp32bulk_bits.txt: the first 16 hex digits of the
SHA-256 of each field's little-endian float64 bytes, on a GB300) hold that apart
from any tolerance.  The inputs are rational functions of integers, so they are the
same bits everywhere; the meshes have shore, dry and deep cells, partly filled
blocks, hanging faces, tide and wall boundaries, friction and tracer diffusion.
"""
import hashlib

import numpy as np
import pytest

from helpers import golden_rows
from paper_2505_18743_gb300 import swdg
from paper_2505_18743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def noise(shape, a, b):
    """integers 0 .. 1008 / 1009, by index"""
    i = np.arange(int(np.prod(shape)), dtype=np.int64)
    return (((i * a + b) ** 2 + 7 * i) % 1009).reshape(shape) / 1009.0


def workload(degree, nx, ny, pix, *, mode=0, tableau=0, f64=False, friction=True, diffusion=False,
             levels=0, seed=1):
    L = 64.0
    if levels:
        mesh, _ = W.forest_mesh(nx, ny, nx * L, ny * L, levels,
                                lambda lev, xc, yc, hx, hy: xc > 0.5 * nx * L, tags=(1, 0, 0, 0))
        npx = pix << (levels - 1)
    else:
        mesh, npx = W.uniform_mesh(nx, ny, nx * L, ny * L, tags=(1, 0, 0, 0)), pix
    m, q = nx * npx, ny * npx
    x = (np.arange(m) + 0.5) / m
    z = 6.0 - 9.0 * x[None, :] + noise((q, m), 31 + seed, 17)
    n, nd = mesh.n, (degree + 1) ** 2
    xc = mesh.x0y0[:, 0:1] / (nx * L)
    zeta = 0.25 * (1.0 - xc) * (noise((n, 1), 7, seed) - 0.5) + 0.02 * (noise((n, nd), 13, seed) - 0.5)
    qx = 0.4 * (noise((n, nd), 5, 3 * seed) - 0.5)
    qy = 0.3 * (noise((n, nd), 11, 5 * seed) - 0.5)
    c = 0.25 + 0.5 * noise((n, nd), 19, seed)
    c[::5] = 0.5  # constant on some cells
    man = 0.02 + 0.02 * noise((n,), 3, seed) if friction else None
    if man is not None:
        man[::7] = 0.0
    return W.Workload(name="bits", degree=degree, mesh=mesh,
                      raster=W.Raster(z if f64 else z.astype(np.float32), 0.0, 0.0, nx * L / m, ny * L / q),
                      zeta=zeta, qx=qx, qy=qy, c=c, tableau=tableau,
                      cfl={1: 0.2, 2: 0.12, 3: 0.08}[degree], subgrid_mode=mode,
                      boundaries=[(0, W.BC_WALL, 0.0, 1.0, 0.0), (1, W.BC_TIDE, 0.4, 44712.0, 0.0)],
                      manning=man, tracer_diffusivity=np.full(n, 0.5) if diffusion else None)


CASES = {
    "r1": dict(degree=1, nx=23, ny=7, pix=8),
    "r2": dict(degree=2, nx=23, ny=7, pix=16),
    "r3": dict(degree=3, nx=21, ny=9, pix=5, f64=True),
    "r3_explicit": dict(degree=3, nx=13, ny=5, pix=16, tableau=1, friction=False),
    "r2_diffusion": dict(degree=2, nx=13, ny=5, pix=11, tableau=3, diffusion=True),
    "r1_points": dict(degree=1, nx=17, ny=6, pix=4, mode=1, f64=True, tableau=2),
    "r3_points": dict(degree=3, nx=11, ny=5, pix=4, mode=1),
    "r2_forest": dict(degree=2, nx=10, ny=4, pix=8, levels=3),
    "r1_forest": dict(degree=1, nx=10, ny=4, pix=8, levels=2, diffusion=True),
    "r2_ensemble": None,
}


def outputs(name):
    """(label, array) of the residual at t = 900 s, the state after three steps, and the
    diagnostics' depth and masses"""
    if CASES[name] is None:
        wls = [workload(2, 9 + 4 * s, 5 + s, 8, seed=s) for s in (1, 2, 3)]
        ctx = swdg.Ensemble.from_workloads(wls, precision=1)
        ctx.set_times(900.0)
        ctx.step(3)
    else:
        ctx = swdg.Context.from_workload(workload(**CASES[name]), precision=1)
        for k, v in ctx.residual(900.0).items():
            yield "residual_" + k, v
        ctx.step(3, -1.0, 900.0)
    for k, v in zip(("zeta", "qx", "qy", "c"), ctx.get_state()):
        yield "state_" + k, v
    ctx.close()


def digest(v):
    return hashlib.sha256(np.ascontiguousarray(v, dtype="<f8").tobytes()).hexdigest()[:16]


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_18743_gb300 import build as B
    B.build()


@pytest.mark.parametrize("name", sorted(CASES))
def test_fp32bulk_bits(name):
    recorded = {r[1]: r[2] for r in golden_rows("fp32bulk_bits.txt") if r[0] == name}
    got = {k: digest(v) for k, v in outputs(name)}
    assert recorded and set(recorded) == set(got)
    assert [k for k in got if got[k] != recorded[k]] == []
