"""The force-field VJP over the sizes where its work split changes: one
reference tile (no split, the gradient written by the pair kernel), ragged
tiles, one and two template points per thread, with template points that
coincide with reference points (their pairs add nothing for p > 1 and the
similarity weight for p = 1).  Tolerance: the relative L2 bar of every force
check against the oracle (float32 pair terms, 1e-5)."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu, check, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


@pytest.mark.parametrize("p", [1.0, 1.5, 2.0, 3.0])
@pytest.mark.parametrize("n,m", [(16, 20), (256, 129), (257, 700), (5003, 333)])
def test_vjp_shapes_match_oracle(n, m, p):
    sc = synth.scale_case()
    X = sc.X[synth.subsample(sc.X, n, n)]
    Y0 = sc.Y0[synth.subsample(sc.Y0, m, m)]
    Y0[: min(n, m) // 4] = X[: min(n, m) // 4]
    d = O.descriptors(X, Y0, O.Params(p=p))
    v = np.random.default_rng(m).normal(size=(m, 3)).astype(np.float32)
    ref = O.force_vjp(Y0, X, d["aY"], d["aX"], d["sigma"], p, 1, v)
    with Gpu(X, Y0, p=p) as g:
        out = torch.full((m, 3), float("nan"), dtype=torch.float32, device="cuda")
        scgr.scgr_force_vjp(g.ctx, torch.from_numpy(v).cuda(), out)
        got = out.cpu().numpy()
    check(f"force VJP, {n} x {m}, p={p:g}: relative L2", rel_l2(got, ref), 1e-5)


def test_vjp_two_points_per_thread():
    """40,000 template points take two points per thread; sampled rows."""
    dc = synth.diff_case(n=40000)
    rng = np.random.default_rng(9)
    a = [np.clip(rng.gamma(1.2, 0.015, size=40000), 0.0, 0.33) for _ in range(2)]
    rows = np.sort(rng.choice(40000, size=48, replace=False))
    rows[0], rows[-1] = 0, 39999
    v = rng.normal(size=(40000, 3)).astype(np.float32)
    ref = O.force_vjp(dc.Y0[rows], dc.X, a[1][rows], a[0], O.sigma_auto(a[0]), 2.0, 1, v[rows])
    with Gpu(dc.X, dc.Y0, p=2.0) as g:
        g.set_curvature(0, a[0])
        g.set_curvature(1, a[1])
        out = torch.full((40000, 3), float("nan"), dtype=torch.float32, device="cuda")
        scgr.scgr_force_vjp(g.ctx, torch.from_numpy(v).cuda(), out)
        got = out.cpu().numpy()
    assert np.isfinite(got).all()
    check("force VJP, 40,000 x 40,000 sampled rows: relative L2", rel_l2(got[rows], ref), 1e-5)
