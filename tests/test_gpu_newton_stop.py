"""Newton's stopping test decides as in FP64: the tolerance at which the continuity
solve of a partly wet cell takes one iteration less is the oracle's, to the accuracy of
the increments themselves (1e-9; an FP32 comparison would be 1e-7 off)."""
import numpy as np
import pytest

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


def _workload(degree, seed):
    wl = W.closed_basin(degree=degree, n=2, pix=16, L=40.0)
    rng = np.random.default_rng(seed)
    z = 2.0 + rng.uniform(-1.0, 1.0, wl.raster.z.shape)
    z[rng.random(z.shape) < 0.2] = -3.0          # pillars, and pixels near the surface
    z[rng.random(z.shape) < 0.2] = 0.05
    wl.raster.z = z
    X, Y = W.nodal_coordinates(wl.mesh, degree)
    wl.zeta = 0.2 + 0.02 * X / 40.0
    wl.qx, wl.qy = 1.5 * np.sin(X / 7.0), 1.5 * np.cos(Y / 9.0)
    wl.tableau, wl.h_lim = 3, 1e-3
    return wl


def threshold(cls, wl, dt):
    """the largest tolerance in [1e-11, 1] at which the result changes, to 1e-11"""
    def result(tol):
        s = cls.from_workload(wl, newton_tol=tol)
        s.step(1, dt, 0.0)
        return np.asarray(s.get_state()[0]).copy()
    lo, hi = 1e-11, 1.0
    top = result(hi)
    assert np.abs(result(lo) - top).max() > 1e-13
    while hi / lo > 1.0 + 1e-11:
        mid = np.sqrt(lo * hi)
        if np.abs(result(mid) - top).max() > 1e-13:
            lo = mid
        else:
            hi = mid
    return hi


@pytest.mark.parametrize("degree, seed", [(2, 2), (2, 3), (3, 4)])
def test_stopping_tolerance(degree, seed):
    wl = _workload(degree, seed)
    got, ref = threshold(swdg.Context, wl, 0.2), threshold(Oracle, wl, 0.2)
    assert abs(got / ref - 1.0) <= 1e-9, (got, ref)
