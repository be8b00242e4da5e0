"""Curvature of nearly and exactly flat kNN neighbourhoods, whose smallest
eigenvalue lies far below the trace: tilted planes (coordinates rounded to
float32 leave about 1e-14), slabs of decreasing thickness, and lines (rank 1).

Bounds against the oracle: 2^-22 relative (four units in the last place of the
float32 curvature) and 2^-48 absolute, for the float64 rounding of a 3 x 3
covariance of unit trace and of its eigenvalues in both codes.  On lines the
middle eigenvalue vanishes too, where the characteristic polynomial determines
its smallest root only to the square root of that rounding: 2^-26 absolute."""
import numpy as np
import pytest

import oracle as O
from paper_1902_01061_gb300 import scgr
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def slab(n, thick, tilt=True):
    rng = np.random.default_rng(n)
    P = rng.uniform(-1, 1, (n, 3)) * [1.0, 1.0, thick]
    if tilt:
        P = P @ np.linalg.qr(rng.standard_normal((3, 3)))[0] + [0.3, -0.2, 0.1]
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("n,k,thick", [(2000, 8, 0.0), (2000, 16, 0.0), (2500, 32, 0.0), (3000, 16, 1e-5), (3000, 32, 1e-4),
                                       (3000, 24, 1e-3), (25000, 16, 1e-6)])
def test_flat_neighbourhoods(n, k, thick):
    P = slab(n, thick)
    with Gpu(P, P, k=k) as g:
        got, nbr = g.curv64(0), g.knn(0)
        np.testing.assert_array_equal(g.curv64(1), got)
    np.testing.assert_allclose(got, O.curvature(P, nbr), rtol=2.0 ** -22, atol=2.0 ** -48)


def test_a_plane_along_the_axes_is_exactly_flat():
    P = slab(1500, 0.0, tilt=False)
    with Gpu(P, P, k=16) as g:
        np.testing.assert_array_equal(g.curv64(0), np.zeros(len(P)))


@pytest.mark.parametrize("grid_min", [None, 0])
def test_lines(grid_min):
    """Three neighbours on each of 200 lines: rank-1 covariances, of which the
    largest root must not be taken for the smallest (curvature 1)."""
    rng = np.random.default_rng(17)
    lines = []
    for q in range(200):  # 5 points on each, 100 apart
        u = rng.normal(size=3)
        lines.append(100.0 * np.array([q % 20, q // 20, 0.0]) + np.outer(np.arange(5.0), u / np.linalg.norm(u)))
    P = np.ascontiguousarray(np.concatenate(lines), np.float32)
    with Gpu(P, P, k=3, tune={} if grid_min is None else {scgr.SCGR_TUNE_KNN_GRID_MIN: grid_min}) as g:
        nbr, got = g.knn(0), g.curv64(0)
    if grid_min == 0:
        np.testing.assert_array_equal(nbr, O.knn(P, 3))
    np.testing.assert_allclose(got, O.curvature(P, nbr), rtol=2.0 ** -22, atol=2.0 ** -26)
