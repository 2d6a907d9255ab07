"""The one-CTA selection of small clouds at its edges: the statistic of a step
against the mean of the ceil(n/100) largest of the same changes (equal to the
rounding of the FP64 sum), and a batch whose clouds lie on both sides of the
line against their own runs (the same bits)."""
import numpy as np
import pytest

import synth
from test_gpu_parity import make_cloud

pytestmark = pytest.mark.gpu


def _handle(dwglib, n, seed):
    p, _, a, eps = make_cloud(n, seed=seed, kind="box")
    h = dwglib.dwg_create(p)
    dwglib.dwg_set_params(h, 0, max(eps, 1e-3), 0.0, 30, 0.1)
    dwglib.dwg_set_update(h, 3, 10, dwglib.DWG_UPDATE_DIRECT)
    dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE, 0.5)
    dwglib.dwg_set_init(h, dwglib.DWG_INIT_GIVEN, 0,
                        synth.random_unit_normals(n, seed=5).astype(np.float32))
    return h


@pytest.mark.parametrize("n", [2, 100, 1023, 1024, 1025, 9217, 16383, 16384, 16385])
def test_statistic(dwglib, oracle_mod, n):
    h = _handle(dwglib, n, n % 97 + 3)
    try:
        dth = np.zeros(n, np.float32)
        for _ in range(2):
            _, stat = dwglib.dwg_step(h, None, None, dth)
            ref = oracle_mod.top1_mean(dth.astype(np.float64))
            assert stat == pytest.approx(ref, rel=1e-12, abs=1e-12)
    finally:
        dwglib.dwg_destroy(h)


@pytest.mark.parametrize("phases", [1, 2])
def test_batch_across_the_line(dwglib, phases):
    sizes = [1000, 16384, 16385, 20000]
    pts = [synth.sphere(n, seed=i)[0] for i, n in enumerate(sizes)]
    P = np.ascontiguousarray(np.vstack(pts))
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    hb = dwglib.dwg_create_batch(P, off)
    try:
        dwglib.dwg_set_batch_mode(hb, phases)
        dwglib.dwg_set_tree(hb, 2, 0.5)
        dwglib.dwg_set_init(hb, 0, 11)
        out = np.zeros_like(P)
        rc, iters = dwglib.dwg_orient_batch(hb, out, len(sizes))
    finally:
        dwglib.dwg_destroy(hb)
    for c, p in enumerate(pts):
        h = dwglib.dwg_create(np.ascontiguousarray(p))
        try:
            # a batch's octree depth goes by each cloud's size, its seed by its place
            depth = min(10, max(5, int(round(0.5 * np.log2(len(p))))))
            dwglib.dwg_set_update(h, depth, 10, dwglib.DWG_UPDATE_LEVELSET)
            dwglib.dwg_set_tree(h, 2, 0.5)
            dwglib.dwg_set_init(h, 0, 11 + c)
            alone = np.zeros_like(p)
            _, it = dwglib.dwg_orient(h, alone)
            assert it == iters[c]
        finally:
            dwglib.dwg_destroy(h)
        assert np.array_equal(out[off[c]:off[c + 1]], alone)
