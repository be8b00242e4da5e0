"""Grid searches at the edges of their geometry, against the oracle's brute
force (indices and keys equal): boxes of subnormal and of very small extent,
whose reciprocals would overflow; thin grids with fewer than k points beyond a
gap of up to tens of thousands of cells; and queries beyond float32's range."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def nearest(g, q):
    idx = torch.empty(len(q), dtype=torch.int32, device="cuda")
    key = torch.empty(len(q), dtype=torch.float32, device="cuda")
    scgr.scgr_nearest(g.ctx, torch.from_numpy(np.ascontiguousarray(q, np.float32)).cuda(), idx, key)
    return idx.cpu().numpy(), key.cpu().numpy()


def brute_nearest(P, q):
    """First of the (key, index) order, every operation rounded on its own."""
    d = q[:, None, :] - P[None, :, :]
    key = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    idx = key.argmin(1)
    return idx, key[np.arange(len(q)), idx]


@pytest.mark.parametrize("extent", [0.0, 1e-45, 1e-39, 5e-39, 1e-31, 2e-30, 1e-12])
def test_boxes_of_tiny_extent(extent):
    P = np.ascontiguousarray(synth.mild(n=1200).X, np.float32)
    P = ((P - P.min(0)) / (P.max(0) - P.min(0)).max()).astype(np.float32) * np.float32(extent)
    with Gpu(P, P, k=16, tune={scgr.SCGR_TUNE_KNN_GRID_MIN: 0}) as g:
        np.testing.assert_array_equal(g.knn(0), O.knn(P, 16))
        q = np.concatenate([P[:50], P[:50] * np.float32(3.0), np.float32([[1, 2, 3], [-1, 0, 1e-20]])])
        idx, key = nearest(g, q)
        want_idx, want_key = brute_nearest(P, q)
        np.testing.assert_array_equal(idx, want_idx)
        np.testing.assert_array_equal(key, want_key)


def gapped(name, n):
    """n points of which 5 lie beyond a gap that is most of the cloud's length."""
    rng = np.random.default_rng(n)
    P = rng.uniform(0.0, 0.1, size=(n, 3))
    P[-5:] = [[1.0, 0, 0], [0.99, 0, 0], [1.0, 0.1, 0.1], [0.985, 0.05, 0.1], [1.0, 0.1, 0]]
    if name == "line":
        P[:, 1:] = 0.25
    elif name == "pole":
        P[:, 1:] *= 0.01
    elif name == "plane":
        P[:, 2] = -1.5
    return np.ascontiguousarray(P, np.float32)


@pytest.mark.parametrize("grid_min", [None, 0])
@pytest.mark.parametrize("name,n,k", [("line", 4000, 16), ("line", 150000, 16), ("pole", 5000, 8), ("pole", 30000, 32),
                                      ("plane", 60000, 16), ("box", 40000, 6)])
def test_few_points_beyond_a_gap(name, n, k, grid_min):
    """All points where the grid's key is asked for and the oracle is quick, else the isolated ones and a sample."""
    P = gapped(name, n)
    rows = np.arange(n) if n <= 5000 else np.concatenate([np.arange(n - 5, n), np.arange(0, n - 5, n // 300)])
    with Gpu(P, P[: max(k, 64)], k=k, tune={} if grid_min is None else {scgr.SCGR_TUNE_KNN_GRID_MIN: grid_min}) as g:
        got = g.knn(0)[rows]
    want = np.concatenate([first_k(P, P[r], k) for r in np.array_split(rows, 1 + len(rows) * n // 20_000_000)])
    if grid_min == 0 or n >= 20000:
        np.testing.assert_array_equal(got, want)
    else:  # near ties may fall either way with the smaller clouds' key (one rounding less)
        np.testing.assert_allclose(dist64(P, rows, got), dist64(P, rows, want), rtol=1e-6)


def first_k(P, q, k):
    d = q[:, None, :] - P[None, :, :]
    key = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    return np.argsort(key, axis=1, kind="stable")[:, :k]


def dist64(P, rows, idx):
    P = P.astype(np.float64)
    return np.linalg.norm(P[idx] - P[rows][:, None, :], axis=2)


@pytest.mark.parametrize("n", [600, 1500, 70000])
def test_queries_beyond_float32_range(n):
    """Where no key is finite the brute-force search (600 points) finds no
    point: index 2^31 - 1, key infinity.  The grid answers the same, whatever
    the finite queries beside them."""
    P = np.ascontiguousarray(synth.mild(n=n).X, np.float32)
    bad = np.float32([[1e30, 0, 0], [0, -3e38, 0], [np.inf, 0, 0], [0, 0, -np.inf], [np.nan, 0, 0], [np.nan] * 3])
    q = np.concatenate([bad, P[:40] + np.float32(0.01), P[:3] * np.float32(1e15), bad])
    with Gpu(P, P[:100], k=8) as g:
        idx, key = nearest(g, q)
    want_idx, want_key = brute_nearest(P, q[6:-6])
    np.testing.assert_array_equal(idx[6:-6], want_idx)
    np.testing.assert_array_equal(key[6:-6], want_key)
    for part in (slice(0, 6), slice(len(q) - 6, len(q))):
        assert np.all(idx[part] == 2**31 - 1) and np.all(np.isposinf(key[part]))


def lattice(n):
    """Points whose neighbour keys tie or nearly tie."""
    g = np.stack(np.meshgrid(*[np.arange(n) * np.float32(0.1)] * 3, indexing="ij"), -1)
    return np.ascontiguousarray(g.reshape(-1, 3), np.float32)


@pytest.mark.parametrize("first,then", [(10**9, 10**9), (10**9, 0), (0, 10**9)])
def test_neighbours_do_not_depend_on_earlier_calls(first, then):
    """After a nearest-point search has built the reference's grid, or with the
    knob changed since the descriptors, the neighbours are those of a context
    that had the knob from the start (the two searches round the key differently)."""
    P = lattice(12)
    with Gpu(P, P, k=16, tune={scgr.SCGR_TUNE_KNN_GRID_MIN: then}) as g:
        want = [g.knn(0), g.knn(1)]
    if then == 0:
        np.testing.assert_array_equal(want[0], O.knn(P, 16))
    with Gpu(P, P, k=16, tune={scgr.SCGR_TUNE_KNN_GRID_MIN: first}) as g:
        nearest(g, P[:64])
        scgr.scgr_set_tuning(g.ctx, scgr.SCGR_TUNE_KNN_GRID_MIN, then)
        scgr.scgr_set_neighbourhood(g.ctx, k=16)
        np.testing.assert_array_equal(g.knn(0), want[0])
        np.testing.assert_array_equal(g.knn(1), want[1])
