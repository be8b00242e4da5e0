"""What a user of this framework has it do, as cases that can be timed and compared.

Every case goes through the public binding (paper_1902_01061_gb300.scgr).  The kinds:

  register     a whole registration: both clouds in, descriptors, iterations, pose and moved cloud out
  descriptors  the one-time descriptor pass of new clouds (k nearest neighbours and curvature)
  forces       one evaluation of the all-pairs force field at the current pose
  potential    the differentiable potential, forward and backward through torch.autograd
  vjp          the vector-Jacobian product of the force field
  mask         the change mask of a registered scan against its reference
  batch        many registrations of uneven sizes in one call
  static       the allocation-free force evaluation on the caller's buffers

Clouds are sampled on the outer surface of a union of ellipsoids, the template being a transformed second
sample with noise and uniform outliers, as in paper_1902_01061_gb300/synth.py but made on the GPU.  Sizes
are those of the repository's benchmark workloads (1,000; 35,000 x 30,800; 50,000; 1,000,000; pairs of
500 to 20,000 points) or odd ones of the same ranges.
"""
import math

import numpy as np
import torch

from paper_1902_01061_gb300 import scgr

G1, ETA0 = 1.0e4, 0.5   # the library's defaults of the Eq. 12 constant and the step fraction


# ---- the cases -------------------------------------------------------------

def listed():
    return [
        # the Fig. 1 setting: a small scan registered over 100 iterations, where each iteration's latency counts
        dict(name="register_1k_p2", kind="register", n=1000, m=1000, k=16, p=2.0, g_mode=1, iters=100, graph=0, radius=0.0),
        # a model-sized scan with the library's default exponent: the pair weights do not depend on the pose
        dict(name="register_35k_p1", kind="register", n=35000, m=30800, k=16, p=1.0, g_mode=1, iters=200, graph=0, radius=0.0),
        # the same scan with the benchmark's exponent: an all-pairs pass in every iteration, replayed from a graph
        dict(name="register_35k_p2", kind="register", n=35000, m=30800, k=16, p=2.0, g_mode=1, iters=20, graph=1, radius=0.0),
        # new small and odd-sized clouds, as a tracker sees them frame by frame
        dict(name="descriptors_5k", kind="descriptors", n=5003, m=4801, k=16, radius=0.0),
        # the largest workload's clouds
        dict(name="descriptors_1m", kind="descriptors", n=1000000, m=1000000, k=16, radius=0.0),
        # the paper's own neighbourhood: every point within the square root of the largest eigenvalue
        dict(name="descriptors_radius_20k", kind="descriptors", n=20011, m=17611, k=16, radius=1.0),
        # one force evaluation of the largest workload's size: the path's throughput
        dict(name="forces_1m_p2", kind="forces", n=1000000, m=1000000, p=2.0, g_mode=1),
        # a general exponent with equal weights (g = s) on odd sizes
        dict(name="forces_20k_p15", kind="forces", n=20011, m=17999, p=1.5, g_mode=0),
        # the differentiable form inside a training step or a pose optimiser
        dict(name="potential_50k_p2", kind="potential", n=50000, m=50000, p=2.0, g_mode=1),
        # back-propagation through the force field
        dict(name="vjp_10k_p2", kind="vjp", n=10007, m=9001, p=2.0, g_mode=1),
        # change detection between two captures that have been registered
        dict(name="mask_300k", kind="mask", n=300000, m=250007),
        # many objects at once, in one CUDA graph
        dict(name="batch_40", kind="batch", pairs=40, lo=500, hi=20000, p=2.0, iters=20, graph=1),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, its sizes spread over the logarithm of their ranges."""
    kind = rng.choice(["register", "register", "descriptors", "descriptors", "forces", "forces", "potential", "vjp",
                       "mask", "batch", "static"])
    if kind == "register":
        p = rng.choice([1.0, 1.0, 2.0, 2.0, 1.5, 3.0])
        n = _log_int(rng, 500, 60000)
        return dict(kind=kind, n=n, m=_about(rng, n), k=rng.choice([8, 16, 16, 24]), p=p, g_mode=rng.choice([0, 1, 1]),
                    iters=rng.choice([10, 20, 50, 100] if n < 8000 or p == 1.0 else [5, 10, 20]),
                    graph=rng.choice([0, 1]), radius=0.0)
    if kind == "descriptors":
        radius = rng.choice([0.0, 0.0, 0.0, 0.5])
        n = _log_int(rng, 500, 40000 if radius else 1000000)
        return dict(kind=kind, n=n, m=_about(rng, n), k=rng.choice([8, 16, 16, 24, 32]), radius=radius)
    if kind == "forces":
        n = _log_int(rng, 500, 400000)
        return dict(kind=kind, n=n, m=_about(rng, n), p=rng.choice([1.0, 1.5, 2.0, 2.0, 3.0]), g_mode=rng.choice([0, 1, 1]))
    if kind == "potential":
        n = _log_int(rng, 1000, 100000)
        return dict(kind=kind, n=n, m=_about(rng, n), p=rng.choice([1.0, 1.5, 2.0, 2.0]), g_mode=rng.choice([0, 1, 1]))
    if kind == "vjp":
        n = _log_int(rng, 1000, 40000)
        return dict(kind=kind, n=n, m=_about(rng, n), p=rng.choice([1.0, 1.5, 2.0, 2.0]), g_mode=rng.choice([0, 1, 1]))
    if kind == "mask":
        n = _log_int(rng, 2000, 500000)
        return dict(kind=kind, n=n, m=_about(rng, n))
    if kind == "batch":
        return dict(kind=kind, pairs=rng.randrange(3, 65), lo=500, hi=_log_int(rng, 1000, 20000), p=rng.choice([1.0, 2.0, 2.0]),
                    iters=rng.choice([5, 10, 20]), graph=rng.choice([0, 1, 1]))
    n = _log_int(rng, 500, 100000)
    return dict(kind=kind, n=n, m=_about(rng, n), p=rng.choice([1.0, 1.5, 2.0, 2.0]), g_mode=rng.choice([0, 1, 1]))


def _about(rng, n):
    return max(64, int(n * rng.uniform(0.7, 1.1)))


# ---- clouds ------------------------------------------------------------------

def _rotation(rng, degrees):
    """Row-vector rotation (y = x @ R) by `degrees` about a random axis."""
    ax = rng.standard_normal(3)
    ax /= np.linalg.norm(ax)
    th = math.radians(degrees)
    K = np.array([[0.0, -ax[2], ax[1]], [ax[2], 0.0, -ax[0]], [-ax[1], ax[0], 0.0]])
    return (np.eye(3) + math.sin(th) * K + (1.0 - math.cos(th)) * (K @ K)).T


class _Surface:
    """The outer surface of a union of `parts` random ellipsoids."""

    def __init__(self, rng, parts):
        self.centres = rng.uniform(-0.5, 0.5, (parts, 3))
        self.axes = rng.uniform(0.3, 1.0, (parts, 3))
        self.rots = np.stack([_rotation(rng, rng.uniform(0.0, 180.0)) for _ in range(parts)])

    def sample(self, gen, n):
        dev = torch.device("cuda")
        put = lambda a: torch.from_numpy(np.ascontiguousarray(a)).to(dev)  # noqa: E731
        centres, axes, rots = put(self.centres), put(self.axes), put(self.rots)
        parts = len(self.axes)
        top = (self.axes.prod(1)[:, None] / self.axes).max(1)          # the largest area element of each ellipsoid
        share = put(top / top.sum()).float()
        got, have = [], 0
        while have < n:
            take = 3 * (n - have) + 1024
            which = torch.multinomial(share, take, replacement=True, generator=gen)
            u = torch.randn((take, 3), device=dev, dtype=torch.float64, generator=gen)
            u /= u.norm(dim=1, keepdim=True)
            a = axes[which]
            element = ((a.prod(1, keepdim=True) / a * u).square().sum(1)).sqrt()
            keep = torch.rand(take, device=dev, dtype=torch.float64, generator=gen) * put(top)[which] < element
            x = torch.einsum("ni,nij->nj", u * a, rots[which]) + centres[which]
            for e in range(parts):
                inside = (((x - centres[e]) @ rots[e].T) / axes[e]).square().sum(1) < 1.0 - 1e-9
                keep &= ~(inside & (which != e))
            x = x[keep]
            got.append(x)
            have += x.shape[0]
        return torch.cat(got)[:n]


def _pair(seed, n, m, degrees=40.0, aligned=False):
    """A reference of n points and a template of m: another sample of the same surface, rotated, scaled and moved
    (unless `aligned`), with noise and 8% uniform outliers in its bounding box.  Float32 [., 3] on the GPU."""
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    surface = _Surface(rng, int(rng.integers(3, 7)))
    x = surface.sample(gen, n)
    out = int(round(0.08 * m))
    y = surface.sample(gen, m - out)
    if not aligned:
        y = 0.9 * y @ torch.from_numpy(_rotation(rng, degrees)).cuda() + torch.from_numpy(rng.uniform(-0.2, 0.2, 3)).cuda()
    y = y + 0.002 * torch.randn(y.shape, device="cuda", dtype=torch.float64, generator=gen)
    lo, hi = y.amin(0), y.amax(0)
    y = torch.cat([y, lo + (hi - lo) * torch.rand((out, 3), device="cuda", dtype=torch.float64, generator=gen)])
    return x.float().contiguous(), y.float().contiguous()


# ---- prepare and run -----------------------------------------------------------

def _registration(case, **more):
    opts = dict(p=case.get("p", 1.0), g_mode=case.get("g_mode", 1), k=case.get("k", 16), use_graph=case.get("graph", 0))
    if case.get("radius", 0.0) > 0.0:
        opts.update(neigh_mode=1, radius_scale=case["radius"])
    opts.update(more)
    return scgr.Registration(**opts)


def _with_clouds(case, seed, **pair):
    x, y = _pair(seed, case["n"], case["m"], **pair)
    reg = _registration(case)
    reg.set_clouds(x, y)
    return reg, x, y


def _pose7(seed):
    rng = np.random.default_rng(seed + 77)
    return np.concatenate([rng.uniform(-0.3, 0.3, 3), rng.uniform(-0.1, 0.1, 3), [1.05]]).astype(np.float32)


def _batch_sizes(case):
    """Log-spaced reference sizes from lo to hi in a random order; each template has up to 15% more points.  The
    sizes belong to the case, not to the seed, so that every pass does the same work."""
    rng = np.random.default_rng(case["pairs"])
    n = np.exp(np.linspace(math.log(case["lo"]), math.log(case["hi"]), case["pairs"])).astype(np.int64)
    rng.shuffle(n)
    return n, (n * rng.uniform(1.0, 1.15, len(n))).astype(np.int64)


def _batch_clouds(case, seed):
    n, m = _batch_sizes(case)
    return [_pair(seed * 1000 + i, int(a), int(b)) for i, (a, b) in enumerate(zip(n, m))]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind in ("register", "descriptors"):
        s["x"], s["y"] = _pair(seed, case["n"], case["m"])
        s["reg"] = _registration(case)
    elif kind == "forces":
        s["reg"], s["x"], s["y"] = _with_clouds(case, seed)
    elif kind == "potential":
        s["reg"], s["x"], s["y"] = _with_clouds(case, seed)
        s["pose"] = torch.from_numpy(_pose7(seed)).requires_grad_(True)
        s["y"].requires_grad_(True)
    elif kind == "vjp":
        s["reg"], s["x"], s["y"] = _with_clouds(case, seed)
        s["v"] = _cotangent(seed, case["m"])
    elif kind == "mask":
        s["reg"], s["x"], s["y"] = _with_clouds(case, seed, aligned=True)
    elif kind == "batch":
        clouds = _batch_clouds(case, seed)
        s["x"] = torch.cat([c[0] for c in clouds])
        s["y"] = torch.cat([c[1] for c in clouds])
        s["xo"] = np.concatenate([[0], np.cumsum([len(c[0]) for c in clouds])]).astype(np.int64)
        s["yo"] = np.concatenate([[0], np.cumsum([len(c[1]) for c in clouds])]).astype(np.int64)
        s["reg"] = _registration(case)
    elif kind == "static":
        s["x"], s["y"] = _pair(seed, case["n"], case["m"])
        s["ax"], s["ay"] = _curvatures(seed, case["n"]), _curvatures(seed + 1, case["m"])
    else:
        raise ValueError(kind)
    return s


def _cotangent(seed, m):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed) + 5)
    return torch.randn((m, 3), device="cuda", dtype=torch.float32, generator=gen)


def _curvatures(seed, n):
    rng = np.random.default_rng(seed + 13)
    return torch.from_numpy(np.clip(rng.gamma(1.2, 0.015, n), 0.0, 0.33)).cuda()


def _matrix(R, t, s):
    """The float32 transform [s R; t] that a caller applies to further points."""
    return np.concatenate([s * np.asarray(R).reshape(3, 3), np.asarray(t).reshape(1, 3)]).astype(np.float32)


MASK_DISTANCE = 0.02


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "register":
        R, t, sc = s["reg"].register(s["x"], s["y"], case["iters"])
        moved = torch.empty_like(s["y"])
        scgr.scgr_get_moved(s["reg"].ctx, moved)
        return dict(pose=_matrix(R, t, sc), moved=moved)
    if kind == "descriptors":
        reg = s["reg"]
        reg.set_clouds(s["x"], s["y"])
        out = {}
        for which, c, label in ((0, s["x"], "x"), (1, s["y"], "y")):
            a = torch.empty(c.shape[0], dtype=torch.float32, device="cuda")
            knn = None if case["radius"] > 0.0 else torch.empty((c.shape[0], case["k"]), dtype=torch.int32, device="cuda")
            scgr.scgr_get_descriptors(reg.ctx, which, knn, a)
            out["a" + label] = a
            if knn is not None:
                out["knn" + label] = knn
        return out
    if kind == "forces":
        return s["reg"].forces()
    if kind == "potential":
        u = scgr.potential(s["pose"], s["y"], s["reg"].ctx)
        gp, gy = torch.autograd.grad(u, (s["pose"], s["y"]))
        return dict(u=u.item(), grad_pose=gp, grad_y=gy)
    if kind == "vjp":
        grad = torch.empty_like(s["v"])
        scgr.scgr_force_vjp(s["reg"].ctx, s["v"], grad)
        return grad
    if kind == "mask":
        m = s["y"].shape[0]
        mask = torch.empty(m, dtype=torch.uint8, device="cuda")
        dist = torch.empty(m, dtype=torch.float32, device="cuda")
        scgr.scgr_change_mask(s["reg"].ctx, MASK_DISTANCE, mask, dist)
        return dict(mask=mask, dist=dist)
    if kind == "batch":
        res = scgr.scgr_batch_run(s["reg"].ctx, s["xo"], s["x"], s["yo"], s["y"], case["iters"])
        return np.stack([_matrix(*r.as_numpy()) for r in res])
    out = torch.empty((case["m"], 4), dtype=torch.float32, device="cuda")
    scgr.scgr_forces_static(s["x"], s["y"], s["ax"], s["ay"], out, p=case["p"], g_mode=case["g_mode"])
    return out


# ---- what a pass cannot do without ----------------------------------------------

def _pair_flops(p):
    """Per pair: difference (3), squared distance (5), similarity (3 + 4), weight (2), sums (7), and the distance
    factor d^(p-1) unless p = 1."""
    return 24 if p == 1.0 else 26


def work(case):
    kind = case["kind"]
    if kind == "batch":
        n, m = (v.astype(float) for v in _batch_sizes(case))
        passes = 1 if case["p"] == 1.0 else case["iters"]
        return dict(bytes=float(12 * (n.sum() + m.sum()) + 48 * len(n)),
                    flops=float((n * m).sum() * _pair_flops(case["p"]) * passes))
    n, m = float(case["n"]), float(case["m"])
    if kind == "register":
        # odd integer exponents need the pairs once, the others in every iteration
        passes = 1 if case["p"] in (1.0, 3.0) else case["iters"]
        return dict(bytes=12 * n + 24 * m + 48, flops=n * m * _pair_flops(case["p"]) * passes + 8 * case["k"] * (n + m))
    if kind == "descriptors":
        if case["radius"] > 0.0:
            # membership of every pair (8 each); the moments of the members are not counted
            return dict(bytes=16 * (n + m), flops=8 * (n * n + m * m))
        return dict(bytes=(16 + 4 * case["k"]) * (n + m), flops=30 * case["k"] * (n + m))
    if kind == "forces":
        return dict(bytes=16 * n + 16 * m + 16 * m, flops=n * m * _pair_flops(case["p"]))
    if kind == "potential":
        return dict(bytes=16 * n + 16 * m + 12 * m, flops=2 * n * m * _pair_flops(case["p"]))
    if kind == "vjp":
        return dict(bytes=16 * n + 16 * m + 24 * m, flops=n * m * 36)
    if kind == "mask":
        return dict(bytes=12 * n + 12 * m + 5 * m, flops=100 * m)
    return dict(bytes=20 * n + 20 * m + 16 * m, flops=n * m * _pair_flops(case["p"]))


# ---- the same in 64 bits ----------------------------------------------------------

MOST_PAIRS = 8.0e10     # pair terms that take about ten seconds in float64
F64 = torch.float64


def _knn(P, k):
    """Indices of the k nearest points of every point (float32 squared distance, self included)."""
    out = []
    for q in P.split(max(1, (1 << 27) // P.shape[0])):
        d = q[:, None, 0] - P[None, :, 0]
        key = d * d
        for c in (1, 2):
            d = q[:, None, c] - P[None, :, c]
            key = key + d * d
        out.append(key.topk(k, dim=1, largest=False).indices)
    return torch.cat(out)


def _surface_variation(C):
    lam = np.linalg.eigvalsh(C.cpu().numpy())
    tr = np.trace(C.cpu().numpy(), axis1=1, axis2=2)
    return torch.from_numpy(np.where(tr > 0, np.maximum(lam[:, 0], 0.0) / np.where(tr > 0, tr, 1.0), 0.0)).cuda()


def _curvature_knn(P, k):
    N = P.double()[_knn(P, k)]
    D = N - N.mean(1, keepdim=True)
    return _surface_variation(torch.einsum("nki,nkj->nij", D, D) / k)


def _curvature_radius(P, scale):
    P64 = P.double()
    c = P64 - P64.mean(0)
    e = float(np.linalg.eigvalsh((c.T @ c / len(c)).cpu().numpy())[-1])
    r2 = torch.tensor(scale * scale * e, dtype=F64).float().item()
    feats = torch.cat([torch.ones_like(c[:, :1]), c, (c[:, :, None] * c[:, None, :]).reshape(-1, 9)], 1)
    out = []
    for q in P.split(max(1, (1 << 26) // P.shape[0])):
        d = P[None, :, 0] - q[:, None, 0]
        key = d * d
        for a in (1, 2):
            d = P[None, :, a] - q[:, None, a]
            key = key + d * d
        S = (key <= r2).double() @ feats
        mean = S[:, 1:4] / S[:, :1]
        out.append((S[:, 4:] / S[:, :1]).reshape(-1, 3, 3) - mean[:, :, None] * mean[:, None, :])
    return _surface_variation(torch.cat(out))


def _curvature(P, case):
    return _curvature_radius(P, case["radius"]) if case.get("radius", 0.0) > 0.0 else _curvature_knn(P, case.get("k", 16))


def _sigma(ax):
    s = float(ax.std(unbiased=False))
    return s if s >= 1e-12 else 1.0


def _rows(Y, X):
    return Y.split(max(1, (1 << 26) // X.shape[0]))


def _pairs(Y, X, ax, ay, sigma, p, g_mode, power):
    """For blocks of template rows: (rows, r_ij components, d^2, g_ij d_ij^power)."""
    at = 0
    for y in _rows(Y, X):
        r = [y[:, None, c] - X[None, :, c] for c in range(3)]
        d2 = r[0] * r[0] + r[1] * r[1] + r[2] * r[2]
        a = ay[at:at + len(y)]
        g = (ax[None, :] - a[:, None]).div_(sigma).square_().neg_().exp_()
        if g_mode == 1:
            g.mul_(ax[None, :]).mul_(a[:, None])
        if power == 1.0:
            g.mul_(d2.sqrt())
        elif power == 2.0:
            g.mul_(d2)
        elif power == 3.0:
            g.mul_(d2).mul_(d2.sqrt())
        elif power != 0.0:
            g.mul_(d2.pow(power / 2.0))
        yield slice(at, at + len(y)), r, d2, g
        at += len(y)


def _forces(Y, X, ax, ay, sigma, p, g_mode):
    out = torch.empty((len(Y), 4), dtype=F64, device="cuda")
    for rows, r, d2, w in _pairs(Y, X, ax, ay, sigma, p, g_mode, p - 1.0):
        for c in range(3):
            out[rows, c] = -(w * r[c]).sum(1)
        out[rows, 3] = w.sum(1)
    return out


def _register(x, y, case):
    """The method of Eq. 5 to Eq. 12 in float64: (4 x 3 transform, moved cloud)."""
    X, Y0 = x.double(), y.double()
    k = case.get("k", 16)
    ax, ay = _curvature_knn(x, k), _curvature_knn(y, k)
    sigma, p, E = _sigma(ax), case["p"], float(case["iters"])
    top = lambda P: np.linalg.eigvalsh(((P - P.mean(0)).T @ (P - P.mean(0)) / len(P)).cpu().numpy())[-1]  # noqa: E731
    eX = top(X)
    Y = Y0.clone()
    R, t, s = np.eye(3), np.zeros(3), 1.0
    fixed = None
    if p == 1.0:    # the weights do not depend on the pose: sum w and sum w X once
        fixed = torch.empty((len(Y), 4), dtype=F64, device="cuda")
        for rows, r, d2, w in _pairs(Y, X, ax, ay, sigma, p, case.get("g_mode", 1), 0.0):
            fixed[rows, 0] = w.sum(1)
            fixed[rows, 1:] = w @ X
    for it in range(case["iters"]):
        if fixed is not None:
            f4 = torch.cat([fixed[:, 1:] - Y * fixed[:, :1], fixed[:, :1]], 1)
        else:
            f4 = _forces(Y, X, ax, ay, sigma, p, case.get("g_mode", 1))
        g = 0.1 + 0.9 / (1.0 + math.exp(-(it - E / 2.0)))
        kappa = ETA0 * g * len(Y) / float(f4[:, 3].sum())
        delta = kappa * f4[:, :3]
        d = delta.mean(0)
        mu = Y.mean(0)
        Yc = Y - mu
        C = ((Yc + delta - d).T @ Yc).cpu().numpy()
        U, S, Vt = np.linalg.svd(C)
        dd = 1.0 if np.linalg.det(Vt.T @ U.T) >= 0 else -1.0
        Rinc = Vt.T @ np.diag([1.0, 1.0, dd]) @ U.T
        c = math.sqrt(eX / top(Y))
        mu_, d_ = mu.cpu().numpy(), d.cpu().numpy()
        t = c * (t - mu_) @ Rinc + mu_ + d_
        U, _, Vt = np.linalg.svd(R @ Rinc)
        R, s = U @ Vt, c * s
        Y = s * Y0 @ torch.from_numpy(R).cuda() + torch.from_numpy(t).cuda()
    return np.concatenate([s * R, t[None]]), Y


def _rodrigues(w):
    th2 = (w * w).sum()
    th = th2.sqrt()
    zero = torch.zeros((), dtype=F64)
    K = torch.stack([torch.stack([zero, -w[2], w[1]]), torch.stack([w[2], zero, -w[0]]), torch.stack([-w[1], w[0], zero])])
    return (torch.eye(3, dtype=F64) + th.sin() / th * K + (1.0 - th.cos()) / th2 * (K @ K)).T


def _pair_terms(case):
    if case["kind"] == "batch":
        n, m = _batch_sizes(case)
        return float((n * m).sum()) * (1 if case["p"] == 1.0 else case["iters"])
    pairs = float(case["n"]) * case["m"]
    if case["kind"] == "register":
        return pairs * (1 if case["p"] == 1.0 else case["iters"]) + float(case["n"]) ** 2
    if case["kind"] == "descriptors":
        return 4.0 * (float(case["n"]) ** 2 + float(case["m"]) ** 2)
    return pairs * (2 if case["kind"] in ("potential", "vjp") else 1) * (2.0 if case.get("p") == 1.5 else 1.0)


def exact(case, seed):
    kind = case["kind"]
    if _pair_terms(case) > MOST_PAIRS:
        return None
    if kind == "batch":
        return np.stack([_register(x, y, dict(case, k=16))[0] for x, y in _batch_clouds(case, seed)])
    x, y = _pair(seed, case["n"], case["m"], aligned=kind == "mask")
    if kind == "register":
        T, moved = _register(x, y, case)
        return dict(pose=T, moved=moved)
    if kind == "descriptors":
        out = dict(ax=_curvature(x, case), ay=_curvature(y, case))
        if case["radius"] == 0.0:
            out.update(knnx=None, knny=None)
        return out
    X, Y0 = x.double(), y.double()
    if kind == "mask":
        dist = torch.empty(len(y), dtype=F64, device="cuda")
        at = 0
        for q in _rows(Y0, X):
            d2 = sum((q[:, None, c] - X[None, :, c]).square() for c in range(3))
            dist[at:at + len(q)] = d2.amin(1).sqrt()
            at += len(q)
        return dict(mask=None, dist=dist)
    p, g_mode = case["p"], case["g_mode"]
    if kind == "static":
        ax, ay = _curvatures(seed, case["n"]), _curvatures(seed + 1, case["m"])
    else:
        if 4.0 * (float(case["n"]) ** 2 + float(case["m"]) ** 2) > 4 * MOST_PAIRS:
            return None
        ax, ay = _curvature_knn(x, 16), _curvature_knn(y, 16)
    sigma = _sigma(ax)
    if kind in ("forces", "static"):
        return _forces(Y0, X, ax, ay, sigma, p, g_mode)
    if kind == "vjp":
        v = _cotangent(seed, case["m"]).double()
        out = torch.empty_like(v)
        for rows, r, d2, w in _pairs(Y0, X, ax, ay, sigma, p, g_mode, p - 1.0):
            rv = sum(r[c] * v[rows, None, c] for c in range(3))
            along = torch.where(d2 > 0, (p - 1.0) * w * rv / torch.where(d2 > 0, d2, 1.0), 0.0)
            W = w.sum(1)
            for c in range(3):
                out[rows, c] = -(W * v[rows, c] + (along * r[c]).sum(1))
        return out
    # potential: U, then its gradient with respect to the moved points (-f) taken through Y = s Y0 R + t
    pose = torch.from_numpy(_pose7(seed)).double().requires_grad_(True)
    R, t, sc = _rodrigues(pose[:3]).cuda(), pose[3:6].cuda(), pose[6].cuda()
    Yleaf = Y0.clone().requires_grad_(True)
    Y = sc * Yleaf @ R + t
    U, G = 0.0, torch.empty_like(Y0)
    for rows, r, d2, w in _pairs(Y.detach(), X, ax, ay, sigma, p, g_mode, p - 1.0):
        U += float((w * d2).sum()) / (p + 1.0)
        for c in range(3):
            G[rows, c] = (w * r[c]).sum(1)
    gp, gy = torch.autograd.grad(Y, (pose, Yleaf), G)
    return dict(u=U, grad_pose=gp, grad_y=gy)
