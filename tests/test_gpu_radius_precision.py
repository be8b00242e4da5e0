"""Radius-neighbourhood curvature where a neighbourhood is small or flat against
the radius, so that sums resolved relative to the radius lose its smallest
eigenvalue: flat clusters a tenth to a ten-thousandth of the radius wide, thin
and exactly planar slabs, sparse neighbourhoods, and coordinates about zero
(whose float32 differences round) and far from it.

Bounds against the oracle: 2^-22 relative (four units in the last place of the
float32 curvature), and 2^-46 absolute for what float64 sums of a few thousand
terms leave of an exact zero."""
import numpy as np
import pytest

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu

RTOL, ATOL = 2.0 ** -22, 2.0 ** -46


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def tilted(rng, x):
    return x @ np.linalg.qr(rng.standard_normal((3, 3)))[0]


def cloud(name, n):
    rng = np.random.default_rng(n)
    P = synth.mild(n=n).X.astype(np.float64)
    if name.startswith("cluster"):   # isolated flat clusters of 40 points, apart from the cloud
        width = float(name[7:])
        for c in range(8):
            at = slice(40 * c, 40 * c + 40)
            patch = rng.uniform(-1, 1, (40, 3)) * [1.0, 1.0, 0.01] * width
            P[at] = tilted(rng, patch) + [4.0 + 3.0 * c, (-1) ** c * 0.3, 0.2]
    elif name == "slab":
        P = tilted(rng, rng.uniform(-1, 1, (n, 3)) * [1.0, 1.0, 0.002])
    elif name == "plane":
        P = tilted(rng, rng.uniform(-1, 1, (n, 3)) * [1.0, 1.0, 0.0])
    elif name == "far":
        P += 300.0
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("name,n,scale", [("cluster0.1", 900, 0.3), ("cluster0.01", 900, 0.3), ("cluster0.0001", 900, 0.3),
                                          ("cluster0.01", 7000, 0.1), ("slab", 800, 0.5), ("slab", 6300, 0.2),
                                          ("plane", 700, 0.4), ("plane", 6200, 0.3), ("mild", 500, 0.5), ("mild", 3000, 0.2),
                                          ("mild", 6500, 0.3), ("far", 1500, 0.3), ("mild", 64, 1.0)])
def test_small_and_flat_neighbourhoods(name, n, scale):
    P = cloud(name, n)
    with Gpu(P, P, neigh_mode=1, radius_scale=scale) as g:
        got, again = g.curv64(0), g.curv64(1)
    want = O.curvature_radius(P, scale)
    np.testing.assert_allclose(got, want, rtol=RTOL, atol=ATOL)
    np.testing.assert_array_equal(got, again)
