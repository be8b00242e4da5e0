"""Radius-neighbourhood curvature of clouds in Morton order, where runs of
points beyond a warp's reach are skipped: sizes that leave ragged runs, tiles
and sort blocks, a small cloud ordered beside a large one, a radius that
reaches everything and one that reaches little, and planar, far-off-centre,
duplicate and clustered clouds.  Bounds: those of the existing radius test
against the oracle (1e-5 relative, 1e-10 absolute); two runs and two equal
clouds give the same bits."""
import numpy as np
import pytest

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def cloud(name, n):
    P = synth.mild(n=n).X
    if name == "planar":
        P[:, 0] = -1.5
    elif name == "far":
        P = P + np.float32(300.0)
    elif name == "twice":
        P[n // 2:] = P[: n - n // 2]
    elif name == "cluster":
        P = P * np.float32(1e-3)
        P[:40] = np.random.default_rng(n).uniform(-5, 5, size=(40, 3))
    elif name == "one":
        P[:] = P[0]
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("name,n,scale", [("plain", 6144, 0.1), ("plain", 6145, 1.0), ("plain", 6177, 20.0),
                                          ("plain", 8193, 0.3), ("planar", 6300, 0.3), ("far", 6400, 0.3),
                                          ("twice", 6501, 0.2), ("cluster", 6200, 0.05)])
def test_ordered_radius_curvature_matches_oracle(name, n, scale):
    P = cloud(name, n)
    Q = synth.mild(n=37).X
    with Gpu(P, Q, neigh_mode=1, radius_scale=scale) as g:
        got, small = g.curv64(0), g.curv64(1)
    with Gpu(P, P, neigh_mode=1, radius_scale=scale) as g:
        again = [g.curv64(0), g.curv64(1)]
    np.testing.assert_allclose(got, O.curvature_radius(P, scale), rtol=1e-5, atol=1e-10)
    np.testing.assert_allclose(small, O.curvature_radius(Q, scale), rtol=1e-5, atol=1e-10)
    np.testing.assert_array_equal(got, again[0])
    np.testing.assert_array_equal(got, again[1])


def test_ordered_radius_curvature_of_coincident_points():
    P = cloud("one", 6150)
    with Gpu(P, P, neigh_mode=1, radius_scale=1.0) as g:
        np.testing.assert_array_equal(g.curv64(0), np.zeros(len(P)))
