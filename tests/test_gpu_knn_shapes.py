"""The grid kNN where its search changes course, against the brute-force
search of the oracle (indices equal): tiny clouds (a grid of one cell), many
exact duplicates (more candidates than a warp keeps, all keys tied), a dense
cluster with far outliers (one crowded cell, cubes that grow over empty
space), a line and a plane, and the smallest and largest k."""
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
    rng = np.random.default_rng(n)
    P = synth.mild(n=n).X
    if name == "duplicates":
        P = np.repeat(P[: max(1, n // 400)], 400, axis=0)[:n]
    elif name == "cluster":
        P = P * np.float32(1e-3)
        P[:20] = rng.uniform(-5, 5, size=(20, 3))
    elif name == "line":
        P = np.outer(np.linspace(0, 1, n), [1.0, 2.0, -0.5])
    elif name == "plane":
        P[:, 1] = 0.0
    elif name == "volume":
        P = rng.uniform(-1, 1, size=(n, 3))
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("name,n,k", [("surface", 32, 32), ("surface", 33, 3), ("surface", 1500, 24), ("surface", 1500, 32),
                                      ("duplicates", 1200, 16), ("duplicates", 900, 32), ("cluster", 1500, 16),
                                      ("line", 700, 16), ("plane", 900, 8), ("volume", 1300, 32)])
def test_grid_knn_edges_match_oracle(name, n, k):
    P = cloud(name, n)
    want = O.knn(P, k)
    with Gpu(P, P, k=k, tune={scgr.SCGR_TUNE_KNN_GRID_MIN: 0}) as g:
        np.testing.assert_array_equal(g.knn(0), want)
        np.testing.assert_array_equal(g.knn(1), want)
