"""The kNN scatter's list scan (32-bit keys, full keys where the tenth and
eleventh agree), its queue of faces without a list (a warp per face) and the
sums' 32-bit tables against the per-thread tree search (knn_lists = 0), which
shares none of the three: the sums are integers, so the normals must be the
same bits."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _cloud(kind, n):
    if kind == "sphere":
        return synth.sphere(n, seed=n)[0]
    if kind == "lattice":  # equal distances everywhere: ties at the tenth neighbour
        k = int(np.ceil(n ** (1 / 3)))
        g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
        return np.ascontiguousarray(g / 8.0, dtype=np.float32)
    if kind == "copies":   # many copies of a few points: zero distances and ties
        p = synth.sphere(max(2, n // 8), seed=3)[0]
        return np.ascontiguousarray(np.resize(p, (n, 3)))
    p = synth.sphere(n, seed=5)[0]  # a dense patch: cells over the list cap
    p[: n // 2] = 0.02 * p[: n // 2] + np.float32([0.7, 0.0, 0.0])
    return np.ascontiguousarray(p)


def _steps(dwglib, p, lists, depth, steps=2):
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_params(h, 0, 0.02, 0.0, 10, 0.1)
        dwglib.dwg_set_update(h, depth, 10, dwglib.DWG_UPDATE_LEVELSET)
        dwglib.dwg_set_tuning(h, knn_lists=lists)
        dwglib.dwg_set_init(h, dwglib.DWG_INIT_RANDOM, 4)
        for _ in range(steps):
            dwglib.dwg_step(h)
        out = np.zeros_like(p)
        dwglib.dwg_get_normals(h, out)
    finally:
        dwglib.dwg_destroy(h)
    return out


@pytest.mark.parametrize("kind", ["sphere", "lattice", "copies", "patch"])
@pytest.mark.parametrize("n,depth", [(2, 3), (9, 4), (10, 4), (11, 2), (16, 5), (33, 6), (257, 5),
                                     (1000, 1), (4096, 7), (20011, 6)])
def test_lists_and_far_queue_equal_the_tree_search(dwglib, kind, n, depth):
    p = _cloud(kind, n)
    a = _steps(dwglib, p, 1, depth)
    b = _steps(dwglib, p, 0, depth)
    assert np.array_equal(a, b), np.abs(a - b).max()
