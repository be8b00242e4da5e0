"""The run, potential, nearest and batch paths at the sizes where their
dispatch or their blocks change.

Tolerances.  Two paths that evaluate the same float32 pair terms differ in the
order of their sums; a row's sums are within C_ROW 2^-24 = 3.8e-6 of their
magnitudes (tests/gpu_helpers.py), so a step's totals are within that of each
other relative to their own magnitudes, and four iterations of a pose update
whose steps are of order one stay within 4 * 3.8e-6 < POSE_TOL = 2e-5 of each
other in the rotation's entries, the translation over the diagonal and the
scale.  Against the oracle the bars are the repository's."""
import numpy as np
import pytest
import torch

import oracle as O
from paper_1902_01061_gb300 import scgr, synth
from tests.gpu_helpers import Gpu, check, rel_l2

pytestmark = pytest.mark.gpu

POSE_TOL = 2e-5
ITERS = 4


@pytest.fixture(scope="module", autouse=True)
def _lib(scgr_lib):
    return scgr_lib


def clouds(n, m):
    case = synth.mild(n=max(n, m))
    return case.X[:n].copy(), case.Y0[synth.subsample(case.Y0, m, 7)]


def same_pose(what, a, b, X):
    Ra, ta, sa = a.as_numpy()
    Rb, tb, sb = b.as_numpy()
    diag = float(np.linalg.norm(X.max(axis=0) - X.min(axis=0)))
    check(f"{what}: rotation entries", np.max(np.abs(Ra - Rb)), POSE_TOL)
    check(f"{what}: translation / diagonal", np.linalg.norm(ta - tb) / diag, POSE_TOL)
    check(f"{what}: scale", abs(sa - sb) / abs(sb), POSE_TOL)


@pytest.mark.parametrize("n,m,p,g_mode", [(1000, 20, 2.0, 1), (300, 512, 1.5, 1), (257, 513, 2.0, 0), (1000, 1024, 2.0, 1),
                                          (2049, 1025, 2.0, 1), (2050, 2048, 1.5, 0), (7680, 540, 2.0, 1)])
def test_one_launch_run_matches_launch_per_pass(n, m, p, g_mode):
    """Small problems run all iterations in one launch (1 to 4 template points
    a lane, the last reference slice ragged); with force timing on, the same
    iterations take two launches each."""
    X, Y0 = clouds(n, m)
    with Gpu(X, Y0, p=p, g_mode=g_mode) as g:
        before = scgr.scgr_launch_count(g.ctx)
        a = g.run(ITERS)
        assert scgr.scgr_launch_count(g.ctx) - before == 1
    with Gpu(X, Y0, p=p, g_mode=g_mode) as g:
        scgr.scgr_set_force_timing(g.ctx, True)
        b = g.run(ITERS)
    same_pose(f"one-launch run, {n} x {m}, p={p:g}", a, b, X)


@pytest.mark.parametrize("n,m,g_mode", [(2100, 2049, 1), (3000, 5003, 0), (20000, 16, 1)])
def test_p1_run_from_moments_matches_recomputed_sums(n, m, g_mode):
    """p = 1: all iterations from the pose-free moments against a force pass
    per iteration."""
    X, Y0 = clouds(n, m)
    out = []
    for reuse in (1, 0):
        with Gpu(X, Y0, p=1.0, g_mode=g_mode, tune={scgr.SCGR_TUNE_REUSE_POSE_FREE: reuse}) as g:
            out.append(g.run(ITERS))
    same_pose(f"p = 1 from moments, {n} x {m}", out[0], out[1], X)


@pytest.mark.parametrize("n,m,p", [(300, 20, 2.0), (257, 129, 1.5), (2600, 1777, 1.0), (600, 4097, 2.0), (700, 4100, 3.0)])
def test_potential_pass_matches_oracle(n, m, p):
    """U and the adjoint from one pair pass: 1 and 2 points a thread (from
    4,096), one and many reference splits, ragged tiles."""
    X, Y0 = clouds(n, m)
    d = O.descriptors(X, Y0, O.Params(p=p))
    pose = np.array([0.3, -0.2, 0.5, 0.1, 0.2, -0.3, 1.2])
    with Gpu(X, Y0, p=p) as g:
        gx = torch.empty((m, 3), dtype=torch.float32, device="cuda")
        U, g7 = scgr.scgr_potential(g.ctx, pose, grad_xyz_out=gx)
        U2, _ = scgr.scgr_potential(g.ctx, pose, want_grad=False)
    Uo, g7o, gyo = O.pose_potential_and_grad(pose, Y0, X, d["aY"], d["aX"], d["sigma"], p, 1)
    check("potential U: relative error", abs(U - Uo) / abs(Uo), 1e-6)
    assert U2 == U
    for sl in (slice(0, 3), slice(3, 6), slice(6, 7)):
        check("pose gradient: block relative L2", rel_l2(g7[sl], g7o[sl]), 1e-4)
    check("template-point gradient: relative L2", rel_l2(gx.cpu().numpy(), gyo), 1e-5)


@pytest.mark.parametrize("levels", [1, 2])
@pytest.mark.parametrize("n,nq", [(1023, 5), (1024, 1), (1024, 130), (5003, 301)])
def test_nearest_on_and_off_the_surface(n, nq, levels):
    """Nearest reference point of queries on the surface, at reference points,
    and far outside the grid: equal to a search over all points under the
    float32 key, ties to the lower index; references below and from the
    grid's smallest size."""
    X, _ = clouds(n, 64)
    rng = np.random.default_rng(n + nq)
    Q = X[rng.integers(0, n, nq)].copy()
    Q[1::3] += rng.normal(scale=0.3, size=Q[1::3].shape).astype(np.float32)
    Q[2::5] *= np.float32(30.0)
    dx, dy, dz = (Q[:, a:a + 1] - X[None, :, a] for a in range(3))
    key = (dx * dx + dy * dy) + dz * dz
    with Gpu(X, X[:64], tune={scgr.SCGR_TUNE_NEAREST_LEVELS: levels}) as g:
        idx = torch.empty(nq, dtype=torch.int32, device="cuda")
        scgr.scgr_nearest(g.ctx, torch.from_numpy(Q).cuda(), idx)
        got = idx.cpu().numpy()
    np.testing.assert_array_equal(got, key.argmin(axis=1))


def test_ragged_batch_matches_single_runs():
    """Pairs of 16 to 3,001 points in one batch (grids of one cell beside large
    ones, clouds of one block and of several) against one run each."""
    sizes = [(16, 16), (33, 17), (3001, 20), (1025, 1024), (40, 2049), (257, 300)]
    pairs = [clouds(n, m) for n, m in sizes]
    off = lambda q: np.concatenate([[0], np.cumsum([len(p[q]) for p in pairs])]).astype(np.int64)
    cat = lambda q: torch.from_numpy(np.concatenate([p[q] for p in pairs])).cuda()
    ctx = scgr.scgr_create(scgr.scgr_default_params(p=2.0))
    try:
        got = scgr.scgr_batch_run(ctx, off(0), cat(0), off(1), cat(1), ITERS)
    finally:
        scgr.scgr_destroy(ctx)
    for (X, Y0), res in zip(pairs, got):
        with Gpu(X, Y0, p=2.0, E=ITERS) as g:
            same_pose(f"batch, {len(X)} x {len(Y0)}", res, g.run(ITERS), X)


@pytest.mark.parametrize("n,m", [(16, 1), (255, 130), (9000, 129), (20011, 300)])
def test_static_forces_split_over_the_reference(n, m):
    """forces_static deals long references of short templates to more blocks;
    rows against the oracle."""
    X, Y = clouds(n, max(m, 16))
    Y = Y[:m].copy()
    rng = np.random.default_rng(n)
    ax = np.clip(rng.gamma(1.2, 0.015, size=n), 0.0, 0.33)
    ay = np.clip(rng.gamma(1.2, 0.015, size=m), 0.0, 0.33)
    out = torch.empty((m, 4), dtype=torch.float32, device="cuda")
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    scgr.scgr_forces_static(dev(X), dev(Y), dev(ax), dev(ay), out, sigma=0.02, p=2.0, g_mode=1)
    f, W = O.forces(Y, X, ay, ax, 0.02, 2.0, 1)
    got = out.cpu().numpy()
    check("forces_static f: relative L2", rel_l2(got[:, :3], f), 1e-5)
    check("forces_static W: relative L2", rel_l2(got[:, 3], W), 1e-5)


@pytest.mark.parametrize("levels", [1, 2])
@pytest.mark.parametrize("name", ["line", "plane", "cluster"])
def test_nearest_through_coarse_cells(name, levels):
    """Grids of many cells on one or two axes, and a dense cluster with far
    points: queries beside, beyond and across the empty cells."""
    rng = np.random.default_rng(8)
    n, nq = 4001, 203
    X = rng.uniform(-1, 1, size=(n, 3))
    if name == "line":
        X = X[:, :1] * np.array([[1.0, 0.0, 0.0]])
    elif name == "plane":
        X[:, 2] = 0.5
    else:
        X *= 1e-3
        X[:7] = rng.uniform(-4, 4, size=(7, 3))
    X = np.ascontiguousarray(X, np.float32)
    Q = rng.uniform(-2, 2, size=(nq, 3)).astype(np.float32)
    Q[::4] = X[rng.integers(0, n, len(Q[::4]))]
    dx, dy, dz = (Q[:, a:a + 1] - X[None, :, a] for a in range(3))
    want = ((dx * dx + dy * dy) + dz * dz).argmin(axis=1)
    with Gpu(X, X[:64], tune={scgr.SCGR_TUNE_NEAREST_LEVELS: levels}) as g:
        idx = torch.empty(nq, dtype=torch.int32, device="cuda")
        scgr.scgr_nearest(g.ctx, torch.from_numpy(Q).cuda(), idx)
        np.testing.assert_array_equal(idx.cpu().numpy(), want)


@pytest.mark.parametrize("want_pose,want_points", [(True, True), (True, False), (False, True)])
def test_potential_autograd_equals_the_entry_point(want_pose, want_points):
    """The gradients that forward forms beside U are the entry point's own bits,
    for each set of inputs that want one, twice over a kept graph; a pose
    changed between forward and backward is still refused."""
    X, Y0 = clouds(700, 650)
    with Gpu(X, Y0, p=2.0) as g:
        pose = torch.tensor([0.3, -0.2, 0.5, 0.1, 0.2, -0.3, 1.2], dtype=torch.float64, requires_grad=want_pose)
        Y = g.Y0.clone().requires_grad_(want_points)
        gx = torch.empty((650, 3), dtype=torch.float32, device="cuda")
        U, g7 = scgr.scgr_potential(g.ctx, pose.detach().numpy(), grad_xyz_out=gx)
        u = scgr.potential(pose, Y, g.ctx)
        assert u.item() == U
        inputs = [t for t, w in ((pose, want_pose), (Y, want_points)) if w]
        want = [t for t, w in ((torch.from_numpy(g7), want_pose), (gx, want_points)) if w]
        for _ in range(2):
            for got, ref in zip(torch.autograd.grad(2.0 * u, inputs, retain_graph=True), want):
                assert torch.equal(got, ref * 2.0)
        if want_pose:
            with torch.no_grad():
                pose += 1.0
            with pytest.raises(RuntimeError):
                torch.autograd.grad(u, inputs)
        with torch.no_grad():
            assert not scgr.potential(pose.detach(), Y, g.ctx).requires_grad
