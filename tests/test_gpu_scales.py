"""Tracers and discharges far outside FP32's range.  The FP64 step is linear in the
concentration, so a tracer scaled by any power of two gives the scaled result (1e-10
of its maximum, the tolerance of the parity tests, against the oracle), although the
mass matrix is inverted in FP32; a continuity residual is linear in the discharges at
rest (1e-12, the residual's)."""
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


def _workload(degree, scale):
    wl = W.closed_basin(degree=degree, n=6, pix=8)
    rng = np.random.default_rng(degree)
    m = wl.raster.z.shape[0]
    x = (np.arange(m) + 0.5) / m
    # an island, so that some cells are partly wet
    wl.raster.z = wl.raster.z - 12.0 * np.exp(-((x[None] - 0.5) ** 2 + (x[:, None] - 0.5) ** 2) / 0.02)
    sh = wl.zeta.shape
    wl.zeta = wl.zeta + 0.02 * rng.standard_normal(sh)
    wl.qx, wl.qy = 0.1 * rng.standard_normal(sh), 0.1 * rng.standard_normal(sh)
    wl.c = rng.uniform(0.2, 1.0, sh) * scale
    return wl


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("power", [-1000, -200, -126, 0, 126, 200, 900])
def test_step_with_scaled_tracer(degree, power):
    s = 2.0 ** power
    one, wl = _workload(degree, 1.0), _workload(degree, s)
    ctx, ora = swdg.Context.from_workload(wl), Oracle.from_workload(one)
    ctx.step(2, -1.0, 0.0)
    ora.step(2, -1.0, 0.0)
    zmax = one.raster.z.reshape(6, 8, 6, 8).max(axis=(1, 3)).ravel()
    wet = np.asarray(ora.get_state()[0]).min(axis=1) + zmax > 1e-3
    for f, a, b in zip(("zeta", "qx", "qy", "c"), ctx.get_state(), ora.get_state()):
        a, b = np.asarray(a), np.asarray(b)
        if f == "c":
            a, b = a[wet] / s, b[wet]
        assert rel_inf(a, b, floor=1.0 if f in ("zeta", "c") else 1e-3) <= 1e-10, f


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("scale", [1e-300, 1e-290, 1e-150])
def test_residual_of_vanishing_discharges(degree, scale):
    wl = _workload(degree, 1.0)
    wl.zeta = np.zeros_like(wl.zeta)
    wl.qx, wl.qy = wl.qx * scale, wl.qy * scale
    got, ref = swdg.Context.from_workload(wl).residual(0.0), Oracle.from_workload(wl).residual(0.0)
    errs = residual_errors({"F": got["F"]}, {"F": ref["F"]})
    assert errs["F"] <= 1e-12
