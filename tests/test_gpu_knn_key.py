"""The neighbours' key at default tuning, on lattices (where near ties are the
rule) and random clouds: below 20,000 points the sums are fused with the
products they add, fma(dz, dz, fma(dx, dx, dy dy)); from 20,000 points on, and
for any cloud that SCGR_TUNE_KNN_GRID_MIN sends to the grid, every operation is
rounded on its own.  Indices are equal to a search with that key."""
import numpy as np
import pytest

from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def lattice(n):
    g = np.stack(np.meshgrid(*[np.arange(n) * np.float32(0.1)] * 3, indexing="ij"), -1)
    return np.ascontiguousarray(g.reshape(-1, 3), np.float32)


def first_k(P, rows, k, fused):
    out = []
    for part in np.array_split(rows, 1 + len(rows) * len(P) // 4_000_000):
        d = P[part][:, None, :] - P[None, :, :]
        x, y, z = d[..., 0], d[..., 1], d[..., 2]
        if fused:  # one rounding of each sum: the extended product and sum are exact or nearly so
            W = np.longdouble
            t = (x.astype(W) * x + (y * y).astype(W)).astype(np.float32)
            key = (z.astype(W) * z + t.astype(W)).astype(np.float32)
        else:
            key = (x * x + y * y) + z * z
        out.append(np.argsort(key, axis=1, kind="stable")[:, :k])
    return np.concatenate(out)


@pytest.mark.parametrize("name,k", [("lattice", 16), ("lattice", 32), ("random", 8), ("random", 24)])
@pytest.mark.parametrize("n", [1728, 19683, 21952])
def test_neighbours_follow_the_stated_key(name, n, k):
    side = round(n ** (1 / 3))
    P = lattice(side) if name == "lattice" else np.ascontiguousarray(synth.mild(n=n).X, np.float32)
    assert len(P) == n
    rows = np.arange(0, n, max(1, n // 500))
    with Gpu(P, P, k=k) as g:
        got, again = g.knn(0), g.knn(1)
    np.testing.assert_array_equal(got, again)
    np.testing.assert_array_equal(got[rows], first_k(P, rows, k, fused=n < 20000))
    with Gpu(P, P, k=k, tune={scgr.SCGR_TUNE_KNN_GRID_MIN: 0}) as g:
        np.testing.assert_array_equal(g.knn(0)[rows], first_k(P, rows, k, fused=False))
