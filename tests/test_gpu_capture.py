"""Nearest-point searches around a caller's CUDA graph: a captured search
answers for the reference of the moment it is replayed, and a search after a
replay that set the reference answers for that reference."""
import numpy as np
import pytest
import torch

from paper_1902_01061_gb300 import scgr, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


N = 3000


def clouds():
    A = np.ascontiguousarray(synth.mild(n=N).X, np.float32)
    return A, np.ascontiguousarray(A[::-1] * np.float32([0.3, 2.0, -1.0]) + np.float32(0.4))


def want(P, q):
    d = q[:, None, :] - P[None, :, :]
    key = (d[..., 0] * d[..., 0] + d[..., 1] * d[..., 1]) + d[..., 2] * d[..., 2]
    idx = key.argmin(1)
    return idx, key[np.arange(len(q)), idx]


class Search:
    """A context on its own stream with queries near and far, and its answers."""

    def __init__(self, q):
        self.q = q
        self.stream = torch.cuda.Stream()
        self.ctx = scgr.scgr_create(scgr.scgr_default_params(k=8), self.stream)
        with torch.cuda.stream(self.stream):
            self.dq = torch.from_numpy(q).cuda()
            self.idx = torch.zeros(len(q), dtype=torch.int32, device="cuda")
            self.key = torch.zeros(len(q), dtype=torch.float32, device="cuda")
            self.x = torch.zeros((N, 3), dtype=torch.float32, device="cuda")
        self.stream.synchronize()

    def put(self, P):
        with torch.cuda.stream(self.stream):
            self.x.copy_(torch.from_numpy(P))
        self.stream.synchronize()

    def nearest(self):
        scgr.scgr_nearest(self.ctx, self.dq, self.idx, self.key)

    def check(self, P):
        self.stream.synchronize()
        idx, key = want(P, self.q)
        np.testing.assert_array_equal(self.idx.cpu().numpy(), idx)
        np.testing.assert_array_equal(self.key.cpu().numpy(), key)

    def capture(self, f):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=self.stream):
            f()
        return g

    def replay(self, g):
        with torch.cuda.stream(self.stream):
            g.replay()
        self.stream.synchronize()

    def __enter__(self):
        return self

    def __exit__(self, *a):
        scgr.scgr_destroy(self.ctx)


def queries(A, B):
    return np.concatenate([A[:200], B[:200], np.float32([[4, 4, 4], [0, -7, 1]])])


@pytest.mark.parametrize("descriptors", [False, True])
def test_captured_search_follows_the_reference(descriptors):
    A, B = clouds()
    with Search(queries(A, B)) as s:
        s.put(A)
        scgr.scgr_set_reference(s.ctx, s.x)
        if descriptors:
            scgr.scgr_set_template(s.ctx, s.x)
            scgr.scgr_compute_descriptors(s.ctx)
        s.nearest()
        s.check(A)
        g = s.capture(s.nearest)
        s.replay(g)
        s.check(A)
        s.put(B)
        scgr.scgr_set_reference(s.ctx, s.x)
        s.replay(g)
        s.check(B)
        s.nearest()
        s.check(B)


@pytest.mark.parametrize("descriptors", [False, True])
def test_search_follows_a_replayed_reference(descriptors):
    A, B = clouds()
    with Search(queries(A, B)) as s:
        def set_up():
            scgr.scgr_set_reference(s.ctx, s.x)
            if descriptors:
                scgr.scgr_set_template(s.ctx, s.x)
                scgr.scgr_compute_descriptors(s.ctx)

        s.put(A)
        set_up()  # sizes the buffers
        g = s.capture(set_up)
        for P in (A, B, A):
            s.put(P)
            s.replay(g)
            for _ in range(2):
                s.nearest()
                s.check(P)


def test_search_between_capture_and_replay_of_the_descriptors():
    A, B = clouds()
    with Search(queries(A, B)) as s:
        s.put(A)
        scgr.scgr_set_reference(s.ctx, s.x)
        scgr.scgr_set_template(s.ctx, s.x)
        scgr.scgr_compute_descriptors(s.ctx)
        s.nearest()
        s.check(A)
        s.put(B)
        scgr.scgr_set_reference(s.ctx, s.x)
        scgr.scgr_set_template(s.ctx, s.x)
        g = s.capture(lambda: scgr.scgr_compute_descriptors(s.ctx))
        s.nearest()
        s.check(B)
        s.replay(g)
        s.nearest()
        s.check(B)
