"""Calls on one cloud refuse a batch handle, which has no points, normals or
octree of its own, and leave it usable."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_calls_on_one_cloud(dwglib):
    d = dwglib
    p = np.ascontiguousarray(synth.sphere(600, seed=1)[0], dtype=np.float32)
    n3, n1 = np.zeros((600, 3), np.float32), np.ones(600, np.float32)
    h = d.dwg_create_batch(p, [0, 200, 600])
    try:
        for call in (lambda: d.dwg_set_weights(h, n1), lambda: d.dwg_set_normals(h, p),
                     lambda: d.dwg_get_normals(h, n3), lambda: d.dwg_eval_gwn(h, p, n1, n3),
                     lambda: d.dwg_knn(h, p, 3, np.zeros((600, 3), np.int64)),
                     lambda: d.dwg_get_leaves(h), lambda: d.dwg_get_corners(h),
                     lambda: d.dwg_profile_step(h), lambda: d.dwg_step(h),
                     lambda: d.dwg_orient(h, n3), lambda: d.dwg_extract_level_set(h),
                     lambda: d.dwg_mlp_features(h, np.zeros((600, 64), np.float32)),
                     lambda: d.dwg_get_tree(h, 600), lambda: d.dwg_set_regularization(h, 1)):
            with pytest.raises(d.DWGError) as e:
                call()
            assert e.value.code == d.DWG_ERR_STATE
        d.dwg_set_params(h, 0, 0.0, 0.0, 2, 0.1)
        d.dwg_orient_batch(h, n3, 2)
        assert np.allclose(np.linalg.norm(n3, axis=1), 1.0, atol=1e-5)
    finally:
        d.dwg_destroy(h)
