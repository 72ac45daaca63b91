"""Residuals on elevations whose gradient is a power of two in the kernels' fixed
point, up to rounding: an affine elevation that rises by a power of two per cell
along one axis (by a third of it along the other, so that neither momentum residual
is round-off) from an offset that is none, against the oracle at the residual
tolerance of the parity tests (1e-12 of a field's maximum)."""
import numpy as np
import pytest

from helpers import residual_errors
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


def _workload(degree, axis, rise, offset):
    n = 8
    wl = W.closed_basin(degree=degree, n=n, pix=4, L=8.0)
    X, Y = W.nodal_coordinates(wl.mesh, degree)
    wl.zeta = offset + rise * (Y + X / 3 if axis else X + Y / 3)  # cells of side 1
    wl.qx, wl.qy = np.zeros_like(X), np.zeros_like(X)
    return wl


@pytest.mark.parametrize("degree", [1, 2, 3])
@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("rise", [1.0, 0.5, -0.25])
def test_affine_elevations(degree, axis, rise):
    for offset in (-0.3, 0.1, 0.2, 1.0 / 3.0):
        wl = _workload(degree, axis, rise, offset)
        errs = residual_errors(swdg.Context.from_workload(wl).residual(0.0),
                               Oracle.from_workload(wl).residual(0.0))
        assert max(errs.values()) <= 1e-12, (offset, errs)


@pytest.mark.parametrize("degree", [1, 2, 3])
def test_affine_elevations_without_allocation(degree):
    from test_zz_no_alloc import run_case
    wls = [_workload(degree, axis, rise, off) for axis in (0, 1)
           for rise, off in ((1.0, -0.3), (0.5, 0.2), (0.25, 0.1))]
    run_case(wls[0], [w.state() for w in wls], 0.0)
