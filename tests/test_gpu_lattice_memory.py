"""The exact path with no scratch for the corners' lattice tasks: the general
evaluator takes the corners, alone and in a batch, and the tasks are made as
soon as there is room.  Both evaluators' corner values agree to 1e-6, so one
iteration's normals do but where a corner within that of the iso-value changes
sides: a few of a thousand points, by the share of one face in many."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

LITTLE = 40_000  # a staged output of 3,000 normals and no more


def _close(a, b):
    d = np.linalg.norm(a - b, axis=1)
    assert np.all(np.isfinite(a)) and np.median(d) <= 1e-5 and d.mean() <= 1e-3


@pytest.mark.parametrize("lam", [0.0, 10.0])
def test_one_cloud(dwglib, lam):
    p, nt = synth.sphere(3000, seed=4)
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_params(h, 1 if lam else 0, 0.02, lam, 1, 0.1)
        dwglib.dwg_set_update(h, 6, 10, dwglib.DWG_UPDATE_LEVELSET)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_ALLPAIRS, 0.5)
        dwglib.dwg_set_init(h, dwglib.DWG_INIT_GIVEN, 0, nt.astype(np.float32))
        dwglib.dwg_get_leaves(h)  # the octree, without the tasks
        dwglib.dwg_set_scratch(h, LITTLE, 0)
        out = [np.zeros((3000, 3), np.float32) for _ in range(3)]
        dwglib.dwg_orient(h, out[0])
        cnt0, iso0 = dwglib.dwg_extract_level_set(h)
        dwglib.dwg_set_scratch(h)
        cnt1, iso1 = dwglib.dwg_extract_level_set(h)
        dwglib.dwg_orient(h, out[1])
        dwglib.dwg_orient(h, out[2])
    finally:
        dwglib.dwg_destroy(h)
    _close(out[0], out[1])
    assert np.array_equal(out[1], out[2])
    assert abs(cnt0 - cnt1) <= 2 + 1e-3 * cnt1 and abs(iso0 - iso1) <= 1e-5 * max(1.0, abs(iso1))


@pytest.mark.parametrize("lanes", [0, 1, 2])
def test_batch(dwglib, lanes):
    sizes = [700, 3000, 1500]
    off = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    p = np.concatenate([synth.sphere(n, seed=n)[0] for n in sizes]).astype(np.float32)
    h = dwglib.dwg_create_batch(p, off)
    try:
        dwglib.dwg_set_batch_mode(h, lanes)
        dwglib.dwg_set_params(h, 0, 0.0, 0.0, 1, 0.1)
        dwglib.dwg_set_init(h, dwglib.DWG_INIT_GAUSS, 1)
        out = [np.zeros_like(p) for _ in range(3)]
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE, 0.5)  # the octrees, without the tasks
        dwglib.dwg_orient_batch(h, out[0], 3)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_ALLPAIRS, 0.5)
        dwglib.dwg_set_scratch(h, LITTLE, 0)
        dwglib.dwg_orient_batch(h, out[0], 3)
        dwglib.dwg_set_scratch(h)
        dwglib.dwg_orient_batch(h, out[1], 3)
        dwglib.dwg_orient_batch(h, out[2], 3)
    finally:
        dwglib.dwg_destroy(h)
    _close(out[0], out[1])
    assert np.array_equal(out[1], out[2])
