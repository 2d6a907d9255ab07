"""Every corner value of the lattice tasks (exact path), through the vertices
of the extracted level set: a vertex lies where w - w_bar changes sign along an
edge of a leaf's tetrahedra, by linear interpolation between the edge's two
corners, so each one shows the values of its own two corners.

With values f0 and f1 at the ends of an edge of length s and an error of d in
each, the crossing moves by at most 2 d s / |f0 - f1|; d is 2e-6 of the
largest |w| (FP32 terms of 1e-7 relative, compensated sums), and float32
positions add 1e-6.  Edges on which that is more than a twentieth of a cell
show nothing and are passed over."""
import numpy as np
import pytest
from scipy.spatial import cKDTree

import synth

pytestmark = pytest.mark.gpu

EDGES = [(a, b) for a in range(8) for b in range(8) if a != b and a & b == a]


def _crossings(L, depth, cb, keys, wc, iso):
    """Crossing points (m, 3) and how far each may be off (m,), the cells' size
    over 20 where it shows nothing; keys: sorted corner keys of wc."""
    S1 = (1 << depth) + 1
    size = 1 << (depth - L[:, 0])
    base = L[:, 1:4] * size[:, None]
    off = np.array([[v >> 0 & 1, v >> 1 & 1, v >> 2 & 1] for v in range(8)])
    X = base[:, None, :] + off[None] * size[:, None, None]
    at = np.searchsorted(keys, (X[..., 0] * S1 + X[..., 1]) * S1 + X[..., 2])
    f = wc[at] - iso
    pos = np.asarray(cb["lo"]) + X * (cb["L"] / (1 << depth))
    h = size * (cb["L"] / (1 << depth))
    d = 2e-6 * max(1.0, np.abs(wc).max())
    pts, tol = [], []
    for a, b in EDGES:
        cut = (f[:, a] > 0) != (f[:, b] > 0)
        fa, fb = f[cut, a], f[cut, b]
        t = fa / (fa - fb)
        pts.append(pos[cut, a] + t[:, None] * (pos[cut, b] - pos[cut, a]))
        s = np.linalg.norm(pos[cut, b] - pos[cut, a], axis=1)
        e = 2.0 * d * s / np.abs(fa - fb) + 1e-6
        tol.append(np.where(e < h[cut] / 20, e, np.inf))
    return np.concatenate(pts), np.concatenate(tol)


def _wrong(V, P, tol):
    """Crossings without a vertex, and vertices without a crossing."""
    sure = np.isfinite(tol)
    miss = (cKDTree(V).query(P[sure])[0] > tol[sure]).sum()
    dist, i = cKDTree(P).query(V)
    return int(miss) + int((dist > tol[i]).sum())


@pytest.mark.parametrize("lam", [0.0, 10.0])
@pytest.mark.parametrize("n,depth", [(5, 3), (127, 4), (129, 6), (1500, 2), (1500, 8), (4100, 6)])
def test_vertices_of_the_level_set(dwglib, oracle_mod, n, depth, lam):
    p = (np.ascontiguousarray(synth.uniform_box(n, [-1] * 3, [1] * 3, seed=n + depth)) if n < 8
         else synth.torus(n, seed=n + depth, noise=0.002)[0])
    n0 = synth.random_unit_normals(n, seed=n).astype(np.float32)
    a = np.full(n, 4.0 / n, np.float32)
    kernel, eps = (1 if lam else 0), 0.05
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_weights(h, a)
        dwglib.dwg_set_params(h, kernel, eps, lam, 3, 0.1)
        dwglib.dwg_set_update(h, depth, 10, dwglib.DWG_UPDATE_LEVELSET)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_ALLPAIRS, 0.5)
        dwglib.dwg_set_normals(h, n0)
        cnt, iso = dwglib.dwg_extract_level_set(h)
        tri = np.zeros((max(cnt, 1), 9), np.float32)
        dwglib.dwg_extract_level_set(h, tri)
    finally:
        dwglib.dwg_destroy(h)
    V = tri[:cnt].reshape(-1, 3).astype(np.float64)
    L = oracle_mod.octree_leaves(p, depth)
    K = oracle_mod.corner_keys(L, depth)
    cb = oracle_mod.cube(p, depth)
    X = oracle_mod.corner_positions(K, depth, cb)
    wc = oracle_mod.gwn(p, n0, a, X, kernel=kernel, eps=eps, lam=lam, grad=False)
    order = np.argsort(K)
    K, wc = K[order], wc[order]
    P, tol = _crossings(L, depth, cb, K, wc, iso)
    assert len(P) and len(V) and np.isfinite(tol).mean() >= 0.9
    assert _wrong(V, P, tol) == 0
    # one corner with its neighbour's value would not pass
    c = int(np.argmax(np.abs(wc - iso)))
    bad = wc.copy()
    bad[c] = 2 * iso - wc[c]
    Pb, tolb = _crossings(L, depth, cb, K, bad, iso)
    assert _wrong(V, Pb, tolb) > 0
