"""w at the octree's leaf corners by the lattice tasks (exact path): the level
set extracted from them against the one from the general evaluator's corner
values (dwg_set_compensation 0 takes it), at the edges of the task layout --
one corner column, one plane, tasks that do not fill a CTA, many CTAs."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _cloud(n, seed):
    if n < 8:
        return np.ascontiguousarray(synth.uniform_box(n, [-1] * 3, [1] * 3, seed=seed))
    return synth.torus(n, seed=seed, noise=0.002)[0]


@pytest.mark.parametrize("lam", [0.0, 10.0])
@pytest.mark.parametrize("n,depth", [(1, 1), (2, 1), (5, 3), (127, 4), (128, 5), (129, 6),
                                     (1500, 2), (1500, 8), (4100, 6)])
def test_level_set_of_the_lattice_tasks(dwglib, oracle_mod, n, depth, lam):
    """Count, vector area, area and enclosed volume of the triangles are sums
    over every leaf, so over every corner value; the iso-value against the
    oracle's w at the points."""
    p = _cloud(n, n + depth)
    n0 = synth.random_unit_normals(n, seed=n).astype(np.float32)
    a = np.full(n, 4.0 / n, np.float32)
    eps = 0.05
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_weights(h, a)
        dwglib.dwg_set_params(h, 1 if lam else 0, eps, lam, 3, 0.1)
        dwglib.dwg_set_update(h, depth, 10, dwglib.DWG_UPDATE_LEVELSET)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_ALLPAIRS, 0.5)
        dwglib.dwg_set_normals(h, n0)
        out = []
        for comp in (1, 0):  # 0: the general evaluator of the uncompensated fold
            dwglib.dwg_set_compensation(h, comp)
            cnt, iso = dwglib.dwg_extract_level_set(h)
            tri = np.zeros((max(cnt, 1), 9), np.float32)
            dwglib.dwg_extract_level_set(h, tri)
            t = tri[:cnt].astype(np.float64).reshape(-1, 3, 3)
            vec = 0.5 * np.cross(t[:, 1] - t[:, 0], t[:, 2] - t[:, 0])
            out.append((cnt, iso, vec.sum(0), np.linalg.norm(vec, axis=1).sum(),
                        np.einsum("ij,ij->", t[:, 0], vec) / 3.0))
    finally:
        dwglib.dwg_destroy(h)
    # both evaluators: FP32 terms of 1e-7 relative, summed over at most n
    # sources; a corner within 1e-6 of the iso-value may change sides and move
    # its cells' triangles by that fraction of a cell
    (c1, i1, v1, a1, o1), (c2, i2, v2, a2, o2) = out
    tol = 1e-4 * max(a1, 1e-3)
    assert abs(i1 - i2) <= 1e-5 * max(1.0, abs(i2))
    assert abs(c1 - c2) <= 2 + 1e-3 * c2
    assert np.abs(v1 - v2).max() <= tol and abs(a1 - a2) <= tol and abs(o1 - o2) <= tol
    # the iso-value is the mean of the oracle's w at the points
    w, _ = oracle_mod.gwn(p, n0, a, p, kernel=1 if lam else 0, eps=eps, lam=lam)
    assert abs(i1 - w.mean()) <= 1e-5 * max(1.0, np.abs(w).max())
