"""Radius-neighbourhood curvature where its sums and splits change: fewer
points than a tile, ragged tiles, several splits of the cloud, every point a
member, a planar and a far-off-centre cloud, duplicates, and very small and
very large coordinates.  Bounds: those of the existing radius test against
the oracle (1e-5 relative, 1e-10 absolute)."""
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
        P[:, 2] = 0.25
    elif name == "far":
        P = P + np.float32(300.0)
    elif name == "twice":
        P[n // 2:] = P[: n - n // 2]
    elif name == "small":
        P = P * np.float32(1e-16)
    elif name == "large":
        P = P * np.float32(1e16)
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("name,n,scale", [("plain", 40, 0.5), ("plain", 255, 0.5), ("plain", 257, 0.2),
                                          ("plain", 1031, 20.0), ("planar", 600, 0.5), ("far", 600, 0.5),
                                          ("twice", 513, 0.3), ("small", 400, 0.5), ("large", 400, 0.5)])
def test_radius_curvature_edges_match_oracle(name, n, scale):
    P = cloud(name, n)
    with Gpu(P, P, neigh_mode=1, radius_scale=scale) as g:
        got = [g.curv64(0), g.curv64(1)]
    want = O.curvature_radius(P, scale)
    np.testing.assert_allclose(got[0], want, rtol=1e-5, atol=1e-10)
    np.testing.assert_array_equal(got[0], got[1])
