"""The work this library is measured on: calls of its public binding, as a
user's program makes them, over the sizes and options of the repository's own
configurations.

A case is a dict of plain values; its "kind" says which call it is:

  eval     dwg_eval_gwn: w (and grad w) of an oriented cloud at query points,
           exact all-pairs or Barnes-Hut
  noalloc  dwg_eval_w_noalloc: w from caller-owned device arrays
  orient   dwg_orient on a handle that is kept (another start or another run
           of the same cloud)
  pipeline a new cloud from upload to oriented normals: dwg_create, area
           weights, initial normals, dwg_orient, dwg_destroy
  warm     the learned start: patch features and the network's forward pass
  train    one training step of that network: gradient and Adam update
  batch    dwg_orient_batch over clouds of uneven size

Inputs are drawn on the GPU from the seed: spheres, tori, bumpy blobs with
outliers and unions of ellipsoids, with analytic normals.  Orientations run a
fixed number of iterations (the tolerance is out of reach), so every pass does
the same work.
"""
import math
import os

import numpy as np
import torch

from paper_2405_13839_gb300 import dwg

DEV = "cuda"
FOUR_PI = 4.0 * math.pi


# ----------------------------------------------------------------------------
# cases
# ----------------------------------------------------------------------------
def listed():
    return [
        # a small model's field at its own size (the 2,000-point sphere): launch latency
        dict(name="eval-sphere-2k", kind="eval", shape="sphere", n=2000, m=2000, queries="near",
             path="allpairs", lam=0.0, grad=True),
        # exact w and gradient at as many places as there are points (the 100k torus)
        dict(name="eval-torus-100k", kind="eval", shape="torus", n=100000, m=100000,
             queries="points", path="allpairs", lam=0.0, grad=True),
        # w alone on a lattice around a mid-sized cloud, screened, ragged sizes: field for meshing
        dict(name="eval-field-50k", kind="eval", shape="blob", n=50001, m=250047,
             queries="lattice", path="allpairs", lam=10.0, grad=False),
        # the far-field path at a lattice around a larger cloud (Barnes-Hut walk)
        dict(name="eval-tree-300k", kind="eval", shape="union", n=300000, m=110592,
             queries="lattice", path="tree", lam=100.0, grad=True),
        # the entry point for callers that own all device memory
        dict(name="noalloc-20k", kind="noalloc", shape="blob", n=20000, m=60001, lam=10.0,
             weights=True),
        # the smallest orientation (2,000-point sphere): many short launches per iteration
        dict(name="orient-sphere-2k", kind="orient", shape="sphere", n=2000, depth=6, knn=10,
             path="allpairs", lam=0.0, theta=0.5, leaf=16, init="random", iters=12),
        # a whole new cloud of 100k points through the exact path, from host memory
        dict(name="pipeline-torus-100k", kind="pipeline", shape="torus", n=100000, depth=8, knn=10,
             path="allpairs", lam=0.0, theta=0.5, leaf=16, init="random", weights="area", iters=8,
             host=True),
        # a whole new cloud of 1M points through the Barnes-Hut path, Voronoi weights, PCA start
        dict(name="pipeline-blob-1m", kind="pipeline", shape="blob", n=1000000, depth=9, knn=10,
             path="tree", lam=100.0, theta=0.4, leaf=32, init="pca", weights="voronoi", iters=8,
             host=False),
        # the largest orientation: iterations of a 4M-point union on a kept handle
        dict(name="orient-union-4m", kind="orient", shape="union", n=4000000, depth=10, knn=10,
             path="tree", lam=100.0, theta=0.6, leaf=16, init="random", iters=3),
        # the learned start of a 200k cloud
        dict(name="warm-200k", kind="warm", shape="blob", n=200000),
        # one step of training that network, with the training script's batch
        dict(name="train-8k", kind="train", b=8192),
        # many clouds at once, most on the exact path, some on the tree
        dict(name="batch-24", kind="batch", clouds=24, lo=3000, hi=100000, lam=10.0, iters=3),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["eval", "eval", "eval", "noalloc", "orient", "orient", "pipeline", "warm",
                       "train", "batch"])
    shape = rng.choice(["sphere", "torus", "blob", "union"])
    lam = rng.choice([0.0, 10.0, 100.0])
    if kind == "eval":
        path = rng.choice(["allpairs", "allpairs", "tree"])
        n = _log_int(rng, 70000, 300000) if path == "tree" else _log_int(rng, 1000, 100000)
        m = _log_int(rng, 500, min(270000, int(2.5e10 / n)))
        return dict(kind=kind, shape=shape, n=n, m=m, path=path, lam=lam,
                    queries=rng.choice(["near", "lattice"] if path == "allpairs" else ["lattice"]),
                    grad=rng.random() < 0.6)
    if kind == "noalloc":
        return dict(kind=kind, shape=shape, n=_log_int(rng, 500, 65536),
                    m=_log_int(rng, 500, 262144), lam=lam, weights=rng.random() < 0.5)
    if kind == "orient":
        tree = rng.random() < 0.5
        n = _log_int(rng, 70000, 2500000) if tree else _log_int(rng, 600, 80000)
        return dict(kind=kind, shape=shape, n=n, depth=_depth(n), knn=10,
                    path="tree" if tree else "allpairs", lam=lam if not tree else 100.0,
                    theta=rng.choice([0.4, 0.5, 0.6]), leaf=rng.choice([16, 32]),
                    init=rng.choice(["random", "gauss", "pca"]), iters=rng.randint(2, 4))
    if kind == "pipeline":
        tree = rng.random() < 0.5
        n = _log_int(rng, 70000, 1000000) if tree else _log_int(rng, 2000, 80000)
        return dict(kind=kind, shape=shape, n=n, depth=_depth(n), knn=10,
                    path="tree" if tree else "allpairs", lam=lam if not tree else 100.0,
                    theta=rng.choice([0.4, 0.5]), leaf=rng.choice([16, 32]),
                    init=rng.choice(["random", "gauss", "pca"]),
                    weights=rng.choice(["area", "voronoi"]), iters=rng.randint(3, 8),
                    host=rng.random() < 0.5)
    if kind == "warm":
        return dict(kind=kind, shape=shape, n=_log_int(rng, 1000, 1000000))
    if kind == "train":
        return dict(kind=kind, b=rng.choice([512, 1000, 4096, 8192, 10007, 16384]))
    return dict(kind=kind, clouds=rng.randint(3, 24), lo=_log_int(rng, 1000, 5000),
                hi=_log_int(rng, 20000, 90000), lam=rng.choice([0.0, 10.0]),
                iters=rng.randint(2, 4))


def _depth(n):
    """Octree depth of a cloud of n points, as the batch handles choose it."""
    return min(10, max(5, int(round(0.5 * math.log2(n)))))


# ----------------------------------------------------------------------------
# inputs
# ----------------------------------------------------------------------------
def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + stream)
    return g


def _rand(g, *shape):
    return torch.rand(*shape, generator=g, device=DEV, dtype=torch.float64)


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device=DEV, dtype=torch.float64)


def _unit(v):
    return v / v.norm(dim=1, keepdim=True).clamp_min(1e-300)


def _rotations(quat):
    """Rotation matrices (k x 3 x 3) of k quaternions."""
    w, x, y, z = _unit(quat).unbind(1)
    return torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                        2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                        2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)],
                       1).view(-1, 3, 3)


def _torus(g, n, R=1.0, r=0.3):
    u = 2 * math.pi * _rand(g, 2 * n + 256)
    v = 2 * math.pi * _rand(g, 2 * n + 256)
    keep = _rand(g, 2 * n + 256) < (R + r * torch.cos(v)) / (R + r)
    u, v = u[keep][:n], v[keep][:n]
    cu, su, cv, sv = torch.cos(u), torch.sin(u), torch.cos(v), torch.sin(v)
    p = torch.stack([(R + r * cv) * cu, (R + r * cv) * su, r * sv], 1)
    return p, torch.stack([cv * cu, cv * su, sv], 1)


def _cloud(shape, n, seed):
    """Points (float32 n x 3), outward normals (float64), mean area weight and softening."""
    g = _gen(seed, 1)
    if shape == "sphere":
        nrm = _unit(_randn(g, n, 3))
        p, area = nrm.clone(), FOUR_PI
    elif shape == "torus":
        p, nrm = _torus(g, n)
        area = FOUR_PI * math.pi * 0.3
        p = p + 0.0005 * _randn(g, n, 3)
    elif shape == "blob":
        # a bumpy closed surface r(u) = 0.45 + bumps, 1 % uniform outliers
        u = _unit(_randn(g, n, 3))
        c = _unit(_randn(g, 12, 3))
        h = 0.05 + 0.15 * _rand(g, 12)
        e = h * torch.exp(6.0 * (u @ c.T - 1.0))
        r = 0.45 + e.sum(1, keepdim=True)
        grad = 6.0 * (e @ c)  # of r over the direction
        grad = grad - (grad * u).sum(1, keepdim=True) * u
        p, nrm = r * u, _unit(u - grad / r)
        k = n // 100
        if k:
            p[:k] = 1.4 * _rand(g, k, 3) - 0.7
        area = FOUR_PI * float((r * r).mean())
    else:
        # a union of 20 ellipsoids and 20 tori of uneven size in the unit cube, 0.1 % noise
        which = torch.randint(0, 40, (n,), generator=g, device=DEV)
        cen = _rand(g, 40, 3)
        axes = 0.04 + 0.11 * _rand(g, 40, 3)
        rot = _rotations(_randn(g, 40, 4))
        u = _unit(_randn(g, n, 3))
        pe, ne = axes[which] * u, _unit(u / axes[which])
        pt, nt = _torus(g, n)
        ring = (which >= 20)[:, None]
        scale = (0.08 + 0.1 * _rand(g, 40, 1))[which]
        loc = torch.where(ring, scale * pt, pe)
        nrm = torch.where(ring, nt, ne)
        R = rot[which]
        p = (R @ loc[:, :, None])[:, :, 0] + cen[which] + 0.001 * _randn(g, n, 3)
        nrm = (R @ nrm[:, :, None])[:, :, 0]
        area = 4.0
    order = torch.randperm(n, generator=g, device=DEV)  # as stored in a file: no order
    p, nrm = p[order].float().contiguous(), nrm[order]
    ext = float((p.amax(0) - p.amin(0)).max())
    return p, nrm, area / n, 0.5 * ext / math.sqrt(n)


def _tilted(nrm, seed):
    """Normals of a nearly converged orientation: a few degrees off, float32."""
    return _unit(nrm + 0.05 * _randn(_gen(seed, 2), *nrm.shape)).float().contiguous()


def _weights(n, mean, seed):
    return (mean * (0.7 + 0.6 * _rand(_gen(seed, 3), n))).float().contiguous()


def _queries(kind, p, m, seed):
    g = _gen(seed, 4)
    if kind == "points":
        return p[:m].clone()
    if kind == "near":
        idx = torch.randint(0, p.shape[0], (m,), generator=g, device=DEV)
        return (p[idx].double() + 0.05 * _randn(g, m, 3)).float().contiguous()
    # the first m nodes of a cubic lattice over the padded bounding box, in raster order
    k = math.ceil(round(m ** (1.0 / 3.0), 6))
    lo, hi = p.amin(0).double(), p.amax(0).double()
    pad = 0.05 * (hi - lo)
    lo, step = lo - pad, (hi - lo + 2 * pad) / max(k - 1, 1)
    i = torch.arange(m, device=DEV)
    ijk = torch.stack([i // (k * k), i // k % k, i % k], 1).double()
    return (lo + ijk * step).float().contiguous()


class _Handle:
    """A library handle that is destroyed with the state that holds it."""

    def __init__(self, h):
        self.h = h

    def __del__(self):
        if self.h is not None:
            dwg.dwg_destroy(self.h)
            self.h = None


def _kernel(lam):
    return dwg.DWG_KERNEL_SCREENED if lam > 0 else dwg.DWG_KERNEL_PLAIN


def _configure(h, case, eps):
    """The settings of an orientation, as a program sets them after dwg_create."""
    dwg.dwg_set_params(h, _kernel(case["lam"]), eps, case["lam"], case["iters"], 1e-6)
    dwg.dwg_set_update(h, case["depth"], case["knn"], dwg.DWG_UPDATE_LEVELSET)
    dwg.dwg_set_convergence(h, dwg.DWG_CONV_MEAN)
    if case["path"] == "tree":
        dwg.dwg_set_tree(h, dwg.DWG_PATH_TREE, case["theta"])
        dwg.dwg_set_tuning(h, tree_leaf=case["leaf"])
    else:
        dwg.dwg_set_tree(h, dwg.DWG_PATH_ALLPAIRS, 0.5)
    dwg.dwg_set_init(h, dict(random=dwg.DWG_INIT_RANDOM, pca=dwg.DWG_INIT_PCA,
                             gauss=dwg.DWG_INIT_GAUSS)[case["init"]], 1)


def _net(seed):
    """The shipped network's parameters, moved a little by the seed."""
    P = np.load(os.path.join(os.path.dirname(os.path.abspath(dwg.__file__)), "warm_start.npy"))
    P = torch.from_numpy(P.astype(np.float32)).to(DEV)
    return (P * (1.0 + 0.01 * _randn(_gen(seed, 5), P.numel()).float())).contiguous()


def _train_inputs(b, seed):
    g = _gen(seed, 6)
    X = torch.zeros(b, 64, device=DEV)
    X[:, :48] = _randn(g, b, 48).float()
    X[:, 48:51] = 0.6 * _randn(g, b, 3).float()
    T = _unit(X[:, 48:51].double() + 0.3 * _randn(g, b, 3)).float().contiguous()
    P = _net(seed)
    m = (0.003 * _randn(g, P.numel())).float()
    v = (1e-5 + 1e-4 * _rand(g, P.numel())).float()
    return X, T, P, m, v


def _batch_sizes(case, seed):
    """Log-uniform sizes, the same for every seed of a case."""
    k = case["clouds"]
    t = [(i + 0.5) / k for i in range(k)]
    order = sorted(range(k), key=lambda i: (i * 7919 + 13) % 104729)
    return [int(round(case["lo"] * (case["hi"] / case["lo"]) ** t[i])) for i in order]


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case)
    if kind == "train":
        X, T, P, m, v = _train_inputs(case["b"], seed)
        s.update(X=X, T=T, P=P, m=m, v=v, g=torch.zeros_like(P))
        return s
    if kind == "batch":
        sizes = _batch_sizes(case, seed)
        kinds = ["sphere", "torus", "blob"]
        pts = torch.cat([_cloud(kinds[i % 3], n, 100 * seed + i)[0] for i, n in enumerate(sizes)])
        off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
        h = _Handle(dwg.dwg_create_batch(pts, off))
        dwg.dwg_set_params(h.h, _kernel(case["lam"]), 0.0, case["lam"], case["iters"], 1e-6)
        dwg.dwg_set_convergence(h.h, dwg.DWG_CONV_MEAN)
        s.update(h=h, k=len(sizes), out=torch.empty_like(pts))
        return s
    p, nrm, a, eps = _cloud(case["shape"], case["n"], seed)
    n = case["n"]
    s["eps"] = eps
    if kind == "eval":
        h = _Handle(dwg.dwg_create(p))
        dwg.dwg_set_weights(h.h, _weights(n, a, seed))
        dwg.dwg_set_params(h.h, _kernel(case["lam"]), eps, case["lam"], 30, 0.1)
        path = dwg.DWG_PATH_TREE if case["path"] == "tree" else dwg.DWG_PATH_ALLPAIRS
        dwg.dwg_set_tree(h.h, path, 0.5)
        dwg.dwg_set_normals(h.h, _tilted(nrm, seed))
        s.update(h=h, q=_queries(case["queries"], p, case["m"], seed),
                 w=torch.empty(case["m"], device=DEV),
                 g=torch.empty(case["m"], 3, device=DEV) if case["grad"] else None)
    elif kind == "noalloc":
        s.update(p=p, nrm=_tilted(nrm, seed), a=_weights(n, a, seed) if case["weights"] else None,
                 q=_queries("near", p, case["m"], seed), w=torch.empty(case["m"], device=DEV))
    elif kind == "orient":
        h = _Handle(dwg.dwg_create(p))
        dwg.dwg_set_weights(h.h, torch.full((n,), a, device=DEV))
        _configure(h.h, case, eps)
        s.update(h=h, out=torch.empty(n, 3, device=DEV))
    elif kind == "pipeline":
        if case["host"]:
            p = p.cpu().numpy()
            s.update(p=p, out=np.empty((n, 3), np.float32), a=np.full(n, a, np.float32))
        else:
            s.update(p=p, out=torch.empty(n, 3, device=DEV), a=torch.full((n,), a, device=DEV))
    elif kind == "warm":
        s.update(h=_Handle(dwg.dwg_create(p)), P=_net(seed), X=torch.empty(n, 64, device=DEV),
                 Y=torch.empty(n, 3, device=DEV))
    else:
        raise ValueError(kind)
    return s


# ----------------------------------------------------------------------------
# one pass
# ----------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "eval":
        dwg.dwg_eval_gwn(s["h"].h, s["q"], s["w"], s["g"])
        return [s["w"], s["g"]] if s["grad"] else [s["w"]]
    if kind == "noalloc":
        dwg.dwg_eval_w_noalloc(s["p"], s["nrm"], s["a"], s["q"], s["w"], _kernel(s["lam"]),
                               s["eps"], s["lam"])
        return [s["w"]]
    if kind == "orient":
        _, iters = dwg.dwg_orient(s["h"].h, s["out"])
        return [s["out"], iters]
    if kind == "pipeline":
        h = dwg.dwg_create(s["p"])
        try:
            if s["weights"] == "voronoi":
                dwg.dwg_voronoi_weights(h, 15)
            else:
                dwg.dwg_set_weights(h, s["a"])
            _configure(h, s, s["eps"])
            _, iters = dwg.dwg_orient(h, s["out"])
        finally:
            dwg.dwg_destroy(h)
        return [s["out"], iters]
    if kind == "warm":
        dwg.dwg_mlp_features(s["h"].h, s["X"])
        dwg.dwg_mlp_forward(s["P"], s["X"], s["Y"])
        return [s["X"], s["Y"]]
    if kind == "train":
        loss = dwg.dwg_mlp_grad(s["P"], s["X"], s["T"], s["g"])
        dwg.dwg_mlp_adam(s["P"], s["g"], s["m"], s["v"], 100, 1e-3)
        return [loss, s["g"], s["P"], s["m"], s["v"]]
    _, iters = dwg.dwg_orient_batch(s["h"].h, s["out"], s["k"])
    return [s["out"], iters]


# ----------------------------------------------------------------------------
# what a pass cannot do without
# ----------------------------------------------------------------------------
def _pair_flops(lam, grad):
    """Floating-point operations of one kernel term (a fused multiply-add is two)."""
    if lam > 0:
        return 41 if grad else 24
    return 33 if grad else 19


def _corners(n, path_depth):
    """Leaf corners of the octree around a surface of n points, at most: its
    occupied cells at the last level grow fourfold per level."""
    return int(min(10.0 * n, 12.0 * 4.0 ** path_depth))


def _iteration(n, depth, tree, lam):
    """Bytes and operations of one iteration: terms at the points (w and grad) and
    at the corners (w); on the tree about 700 terms per query."""
    c = _corners(n, depth)
    terms = 700 if tree else n
    return 40.0 * n + 36.0 * c, float(terms) * (n * _pair_flops(lam, True) + c * _pair_flops(lam, False))


def work(case):
    kind = case["kind"]
    if kind == "train":
        return {"bytes": 4.0 * (67 * case["b"] + 8 * 12675), "flops": 6.0 * 12480 * case["b"]}
    if kind == "batch":
        b = f = 0.0
        for n in _batch_sizes(case, 0):
            x, y = _iteration(n, _depth(n), n > 65536, case["lam"])
            b, f = b + 24.0 * n + x * case["iters"], f + y * case["iters"]
        return {"bytes": b, "flops": f}
    n = case["n"]
    if kind in ("eval", "noalloc"):
        m, grad = case["m"], case.get("grad", False)
        terms = 1500 if case.get("path") == "tree" else n
        return {"bytes": 28.0 * n + (28.0 if grad else 16.0) * m,
                "flops": float(terms) * m * _pair_flops(case["lam"], grad)}
    if kind in ("orient", "pipeline"):
        b, f = _iteration(n, case["depth"], case["path"] == "tree", case["lam"])
        return {"bytes": 28.0 * n + b * case["iters"], "flops": f * case["iters"]}
    return {"bytes": (12.0 + 2 * 256.0 + 12.0) * n + 4 * 12675, "flops": 2.0 * 12480 * n}


# ----------------------------------------------------------------------------
# the same in 64 bits
# ----------------------------------------------------------------------------
def _exact_field(p, mom, q, eps, lam, grad):
    """w and grad w of Eq. 2/3 or Eq. 5 (softened), sources equal to the query left out."""
    p, mom, q = p.double(), mom.double(), q.double()
    o = p.mean(0)
    p, q = p - o, q - o
    s = math.sqrt(lam)
    pp, pm = (p * p).sum(1), (p * mom).sum(1)
    ws, gs = [], []
    step = max(1, (1 << 26) // p.shape[0])
    for i in range(0, q.shape[0], step):
        a = q[i:i + step]
        rr = ((a * a).sum(1, keepdim=True) + pp - 2.0 * (a @ p.T)).clamp_min_(0.0)
        far = (rr > 1e-13).double()
        rr += eps * eps
        inv = rr.rsqrt()
        md = pm - a @ mom.T
        i2 = inv * inv
        e = torch.exp(-s * rr * inv) * far if lam > 0 else far
        k = e * i2 * (inv + s)  # F / rho^3
        ws.append((k * md).sum(1))
        if grad:
            c = md * i2 * (3.0 * k + s * s * e * inv)
            gs.append(c @ p - a * c.sum(1, keepdim=True) - k @ mom)
    return [torch.cat(ws)] + ([torch.cat(gs)] if grad else [])


def _exact_train(case, seed):
    X, T, P, m, v = (t.double() for t in _train_inputs(case["b"], seed))
    P.requires_grad_(True)
    parts, o = [], 0
    for rows, cols in ((64, 64), (64, 64), (64, 64), (3, 64)):
        parts.append((P[o:o + rows * cols].view(rows, cols), P[o + rows * cols:o + rows * cols + rows]))
        o += rows * cols + rows
    y = X
    for i, (W, b) in enumerate(parts):
        y = y @ W.T + b
        if i < 3:
            y = torch.relu(y)
    loss = ((y - T) ** 2).sum() / case["b"]
    loss.backward()
    g = P.grad
    m = 0.9 * m + 0.1 * g
    v = 0.999 * v + 0.001 * g * g
    new = P.detach() - 1e-3 * (m / (1 - 0.9 ** 100)) / ((v / (1 - 0.999 ** 100)).sqrt() + 1e-8)
    return [float(loss.detach()), g, new, m, v]


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        return _exact_train(case, seed)
    if kind not in ("eval", "noalloc"):
        return None  # discrete steps (faces, nearest points) between the sums: no plain form
    p, nrm, a, eps = _cloud(case["shape"], case["n"], seed)
    if kind == "noalloc" and not case["weights"]:
        wt = torch.ones(case["n"], 1, device=DEV, dtype=torch.float64)
    else:
        wt = _weights(case["n"], a, seed).double()[:, None]
    mom = _unit(_tilted(nrm, seed).double()) * wt / FOUR_PI
    q = _queries(case["queries"] if kind == "eval" else "near", p, case["m"], seed)
    eps = float(np.float32(eps))
    return _exact_field(p, mom, q, eps, float(np.float32(case["lam"])), case.get("grad", False))
