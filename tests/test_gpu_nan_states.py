"""The positivity step of a state that holds NaN or infinite discharges, or NaN
elevations: a face point whose one side has no wave speed takes the other side's, as
the oracle does (1e-13)."""
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


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("where", ["fine", "coarse", "one"])
@pytest.mark.parametrize("field, value", [(0, np.nan), (1, np.nan), (2, np.nan), (1, -np.nan), (2, -np.nan),
                                          (1, np.inf), (2, np.inf)])
def test_positivity_step(degree, field, where, value):
    mesh, level = W.forest_mesh(4, 2, 400.0, 200.0, 2, lambda lev, xc, yc, hx, hy: xc > 200.0)
    n, nd = mesh.n, (degree + 1) ** 2
    rng = np.random.default_rng(1)
    u = [0.01 * rng.standard_normal((n, nd)), 0.1 * rng.standard_normal((n, nd)),
         0.1 * rng.standard_normal((n, nd)), np.ones((n, nd))]
    cells = {"fine": level == 1, "coarse": level == 0, "one": np.arange(n) == n // 2}[where]
    u[field][cells] = value
    wl = W.Workload("nan", degree, mesh, W.Raster(np.full((16, 32), 5.0), 0.0, 0.0, 12.5, 12.5), *u)
    got, ref = swdg.Context.from_workload(wl).cfl_dt(0.0), Oracle.from_workload(wl).cfl_dt(0.0)
    assert abs(got - ref) <= 1e-13 * ref
