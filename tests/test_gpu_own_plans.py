"""The force VJP and the potential choose their grids from the clouds' sizes:
the bits do not depend on what the context held before nor on the force
kernel's tuning knobs."""
import numpy as np
import pytest
import torch

from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


KNOBS = [{}, {scgr.SCGR_TUNE_FORCE_SPLITS: 1}, {scgr.SCGR_TUNE_FORCE_SPLITS: 64},
         {scgr.SCGR_TUNE_FORCE_P: 4, scgr.SCGR_TUNE_FORCE_TPB: 128}]


def clouds(n, m):
    return np.ascontiguousarray(synth.mild(n=n).X, np.float32), np.ascontiguousarray(synth.mild(n=m, seed=5).Y0, np.float32)


def vjp(g, m):
    v = torch.from_numpy(np.random.default_rng(m).standard_normal((m, 3)).astype(np.float32)).cuda()
    out = torch.empty_like(v)
    scgr.scgr_force_vjp(g.ctx, v, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("n,m,p", [(900, 700, 2.0), (5003, 4801, 1.0), (5003, 4801, 1.5), (3000, 9000, 2.0), (257, 70, 3.0)])
def test_vjp_bits_do_not_depend_on_history_or_knobs(n, m, p):
    X, Y = clouds(n, m)
    got = []
    for tune in KNOBS:
        with Gpu(X, Y, p=p, tune=tune) as g:
            got.append(vjp(g, m))
    big = clouds(12000, 12000)
    with Gpu(*big, p=p) as g:  # a context whose buffers have grown
        vjp(g, 12000)
        g.m = m
        scgr.scgr_set_reference(g.ctx, torch.from_numpy(X).cuda())
        scgr.scgr_set_template(g.ctx, torch.from_numpy(Y).cuda())
        scgr.scgr_compute_descriptors(g.ctx)
        got.append(vjp(g, m))
    assert np.isfinite(got[0]).all() and np.abs(got[0]).max() > 0
    for other in got[1:]:
        np.testing.assert_array_equal(other, got[0])


@pytest.mark.parametrize("n,m,p", [(900, 700, 2.0), (5003, 4801, 1.0), (5003, 4801, 1.5), (3000, 9000, 2.0), (257, 70, 3.0)])
def test_potential_bits_do_not_depend_on_the_force_knobs(n, m, p):
    X, Y = clouds(n, m)
    pose = np.array([0.2, -0.1, 0.3, 0.05, 0.0, -0.1, 1.05])
    got = []
    for tune in KNOBS:
        with Gpu(X, Y, p=p, tune=tune) as g:
            gx = torch.empty((m, 3), dtype=torch.float32, device="cuda")
            U0, _ = scgr.scgr_potential(g.ctx, pose, want_grad=False)
            U, g7 = scgr.scgr_potential(g.ctx, pose, grad_xyz_out=gx)
            got.append((U0, U, g7, gx.cpu().numpy()))
    assert np.isfinite(got[0][3]).all() and got[0][1] > 0
    for other in got[1:]:
        for a, b in zip(other, got[0]):
            np.testing.assert_array_equal(a, b)
