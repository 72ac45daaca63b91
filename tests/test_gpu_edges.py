"""Residual, step and FP32-bulk residual against the oracle at the edges of the
kernels' work split: cell counts that leave lanes, warps and blocks partly
filled (a warp holds 1, 2 or 4 cells, by degree), and pixel counts from one per
cell to the largest.  Tolerances as in the parity and FP32-bulk tests (1e-12 of
a residual field's maximum, 1e-10 of a state's, 1e-5 for FP32 terms; the FP32
path's continuity and tracer residuals contain the FP32 discharges and share the
latter).  The tracer of a cell without water is 0 / 0 up to round-off and is not
compared."""
import numpy as np
import pytest

from helpers import rel_inf, residual_errors
from oracle.oracle import Oracle
from paper_2505_18743_gb300 import swdg
from paper_2505_18743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from oracle import oracle
    from paper_2505_18743_gb300 import build as B
    B.build()
    oracle.build()


def _workload(degree, n, pix):
    wl = W.closed_basin(degree=degree, n=n, pix=pix)
    rng = np.random.default_rng(10 * degree + n)
    m = wl.raster.z.shape[0]
    x = (np.arange(m) + 0.5) / m
    # an island that rises above the water in the middle of the basin
    wl.raster.z = wl.raster.z - 12.0 * np.exp(-((x[None] - 0.5) ** 2 + (x[:, None] - 0.5) ** 2) / 0.02)
    sh = wl.zeta.shape
    wl.zeta = wl.zeta + 0.02 * rng.standard_normal(sh)
    wl.qx, wl.qy = 0.1 * rng.standard_normal(sh), 0.1 * rng.standard_normal(sh)
    wl.c = rng.uniform(0.2, 1.0, sh)
    return wl


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("n, pix", [(1, 4), (3, 1), (5, 3), (7, 32), (13, 5)])
def test_residual_and_step_at_partial_fills(degree, n, pix):
    wl = _workload(degree, n, pix)
    ctx, ora = swdg.Context.from_workload(wl), Oracle.from_workload(wl)
    errs = residual_errors(ctx.residual(0.0), ora.residual(0.0))
    assert max(errs.values()) <= 1e-12, errs
    bulk = swdg.Context.from_workload(wl, precision=1)
    errs = residual_errors(bulk.residual(0.0), ora.residual(0.0))
    assert max(errs.values()) <= 1e-5, errs
    ctx.step(1, -1.0, 0.0)
    ora.step(1, -1.0, 0.0)
    new, ref = ctx.get_state(), ora.get_state()
    zmax = wl.raster.z.reshape(n, pix, n, pix).max(axis=(1, 3)).ravel()
    wet = np.asarray(ref[0]).min(axis=1) + zmax > 1e-3
    assert wet.any()
    for f, a, b in zip(("zeta", "qx", "qy", "c"), new, ref):
        if f == "c":
            a, b = np.asarray(a)[wet], np.asarray(b)[wet]
        assert rel_inf(a, b, floor=1.0 if f in ("zeta", "c") else 1e-3) <= 1e-10, f
