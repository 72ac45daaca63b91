"""Consistency with continuity of the FP64 residual: with c = 1 the tracer residual is
the continuity residual.  The two are formed apart (the tracer's point values are
products of digit pairs), and may differ by FP64's last place: 2^-53 of F in the root
mean square, 2^-51 of its maximum anywhere."""
import numpy as np
import pytest

from paper_2505_18743_gb300 import swdg
from paper_2505_18743_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _build():
    from paper_2505_18743_gb300 import build as B
    B.build()


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("n, pix", [(6, 4), (11, 3)])
def test_tracer_residual_of_unit_concentration(degree, n, pix):
    wl = W.closed_basin(degree=degree, n=n, pix=pix)
    rng = np.random.default_rng(degree + n)
    X, Y = W.nodal_coordinates(wl.mesh, degree)
    wl.c = np.ones_like(X)
    wl.qx = X / 1000.0 - 0.5 + 1e-3 * rng.standard_normal(X.shape)
    wl.qy = Y / 1000.0 - 0.5 + 1e-3 * rng.standard_normal(X.shape)
    r = swdg.Context.from_workload(wl).residual(0.0)
    d = np.abs(r["R"] - r["F"])
    assert d.max() <= 2.0 ** -51 * np.abs(r["F"]).max()
    assert np.sqrt((d ** 2).mean() / (r["F"] ** 2).mean()) <= 2.0 ** -53
