"""Grid searches at the edges of their geometry, against the oracle's brute
force (indices and keys equal): boxes of subnormal and of very small extent,
whose reciprocals would overflow."""
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
