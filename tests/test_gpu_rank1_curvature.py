"""Curvature of collinear neighbourhoods, whose covariance has rank 1 (its
smallest eigenvalue is 0 and the characteristic polynomial's coefficients are
rounding), against the oracle: sparse clouds whose radius neighbourhoods hold
two points.  Bounds: those of the existing radius test (1e-5 relative, 1e-10
absolute)."""
import numpy as np
import pytest

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


@pytest.mark.parametrize("n,scale", [(2000, 0.05), (2000, 0.1), (500, 0.2)])
def test_radius_neighbourhoods_of_two_points(n, scale):
    P = np.ascontiguousarray(synth.mild(n=n).X, np.float32)
    want = O.curvature_radius(P, scale)
    with Gpu(P, P, neigh_mode=1, radius_scale=scale) as g:
        np.testing.assert_allclose(g.curv64(0), want, rtol=1e-5, atol=1e-10)

