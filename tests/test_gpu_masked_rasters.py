"""Rasters whose dry pixels lie far above the water: land or no-data values (-9999,
-1e10, the lowest FP32 value, -infinity) and cliffs beside a film of water.  A dry
pixel adds nothing to a sub-grid sum, so these meet the tolerances of any other
raster: 1e-12 of a residual field's maximum, 1e-10 of a state's, 1e-5 in FP32-bulk,
1e-11 for the residual's pull-back, 1e-9 for a step's."""
import numpy as np
import pytest

from helpers import rel_inf, residual_errors
from oracle.oracle import Oracle
from oracle.torch_residual import TorchResidual, residual_vjp
from oracle.torch_step import TorchStep, step_vjp
from paper_2505_18743_gb300 import swdg
from paper_2505_18743_gb300 import workloads as W

pytestmark = pytest.mark.gpu

LAND = {"9999": -9999.0, "1e10": -1e10, "lowest": -3.4028234663852886e38, "inf": -np.inf}


@pytest.fixture(scope="module", autouse=True)
def _build():
    from oracle import oracle
    from paper_2505_18743_gb300 import build as B
    B.build()
    oracle.build()


def masked(degree, land, dtype=np.float64, n=6, pix=8):
    """a basin with 3 x 3 pixel blocks of land"""
    wl = W.closed_basin(degree=degree, n=n, pix=pix)
    rng = np.random.default_rng(degree)
    z = np.array(wl.raster.z)
    for j, i in ((5, 5), (13, 22), (30, 9), (33, 40), (24, 24)):
        z[j:j + 3, i:i + 3] = land
    wl.raster.z = z.astype(dtype)
    sh = wl.zeta.shape
    wl.zeta = wl.zeta + 0.02 * rng.standard_normal(sh)
    wl.qx, wl.qy = 0.1 * rng.standard_normal(sh), 0.1 * rng.standard_normal(sh)
    wl.c = rng.uniform(0.2, 1.0, sh)
    wl.manning = np.full(wl.mesh.n, 0.03)
    return wl


def cliff(degree, height, base=0.0, dtype=np.float64):
    """a film of 0.1 mm at the foot (or, base < 0, on top) of a cliff, beside deeper water"""
    wl = masked(degree, -9999.0, dtype)
    m = wl.raster.z.shape[0]
    wl.raster.z = np.full((m, m), base)
    wl.raster.z[:, : m // 2] += 0.5
    for j, i in ((5, 5), (13, 26), (30, 9), (33, 40), (24, 24)):
        wl.raster.z[j:j + 3, i:i + 3] = base - height
    wl.raster.z = wl.raster.z.astype(dtype)
    wl.zeta = np.full_like(wl.zeta, 1e-4) - base
    wl.qx, wl.qy = 1e-5 * wl.qx, 1e-5 * wl.qy
    wl.eps_vel = 1e-5
    wl.h_lim = 1e-6
    return wl


def check(wl, tol=1e-12, state_tol=1e-10):
    ctx, ora = swdg.Context.from_workload(wl), Oracle.from_workload(wl)
    errs = residual_errors(ctx.residual(0.0), ora.residual(0.0))
    assert max(errs.values()) <= tol, errs
    ctx.step(1, -1.0, 0.0)
    ora.step(1, -1.0, 0.0)
    for f, a, b in zip(("zeta", "qx", "qy", "c"), ctx.get_state(), ora.get_state()):
        assert rel_inf(a, b, floor=1e-3) <= state_tol, f


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("land", sorted(LAND))
def test_land_values(degree, dtype, land):
    wl = masked(degree, LAND[land], dtype)
    check(wl)
    bulk = swdg.Context.from_workload(wl, precision=1)
    errs = residual_errors(bulk.residual(0.0), Oracle.from_workload(wl).residual(0.0))
    assert max(errs.values()) <= 1e-5, errs
    bulk.step(1, -1.0, 0.0)


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("height", [300.0, 2000.0])
def test_cliffs_beside_a_film(degree, dtype, height):
    check(cliff(degree, height, dtype=dtype))


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("land", sorted(LAND))
def test_land_values_without_allocation(degree, land):
    from test_zz_no_alloc import perturbed, run_case
    wl = masked(degree, LAND[land])
    run_case(wl, [wl.state(), perturbed(wl.state(), 3)], 0.0)
    film = cliff(degree, 2000.0)
    run_case(film, [film.state()], 0.0)


def test_land_values_on_a_forest():
    """hanging faces: the half strips have no bounds of their own"""
    wl = masked(2, -3.4e38)
    mesh, _ = W.forest_mesh(3, 3, 1000.0, 1000.0, 2, lambda lev, xc, yc, hx, hy: xc > 500.0)
    sub = W.Workload(**{**wl.__dict__, "mesh": mesh})
    rng = np.random.default_rng(5)
    sh = (mesh.n, 9)
    sub.zeta = 0.05 * rng.standard_normal(sh)
    sub.qx, sub.qy = 0.1 * rng.standard_normal(sh), 0.1 * rng.standard_normal(sh)
    sub.c, sub.manning = rng.uniform(0.2, 1.0, sh), np.full(mesh.n, 0.03)
    check(sub)


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("land", ["9999", "1e10", "lowest"])
def test_pull_backs_with_land(degree, land):
    wl = masked(degree, LAND[land])
    wl.tableau, wl.h_lim = 0, 1e-3
    n, nd = wl.mesh.n, (degree + 1) ** 2
    rng = np.random.default_rng(7)
    cot = [rng.standard_normal((n, nd)) for _ in range(6)]
    tr = TorchResidual(wl.mesh, wl.raster, degree, 0, wl.g, wl.eps_vel, wl.boundaries, None)
    ref = residual_vjp(tr, wl.state(), wl.manning, np.zeros(n), cot, 0.0)
    ctx = swdg.Context.from_workload(wl)
    got = ctx.residual_vjp(cot, 0.0)
    # (the bottom is flat between its steps, where the offset's derivative is one-sided)
    for key, r in zip(("zeta", "qx", "qy", "c", "manning"), ref):
        assert rel_inf(got[key], r) <= 1e-11, key
    dt = 0.05
    ref = step_vjp(TorchStep(wl), wl.state(), wl.manning, np.zeros(n), cot[:4], 0.0, dt, 1)
    ctx.step_record(dt, 0.0)
    got = ctx.step_vjp(cot[:4])
    for key, r in zip(("zeta", "qx", "qy", "c", "manning"), ref):
        assert rel_inf(got[key], r) <= 1e-9, key
