"""dwg_eval_gwn on the Barnes-Hut path under the group test evaluates each call
through interaction lists of its own.  A query's terms depend on its group of
64 only, so a call with more queries behind it, or cut into work items of
another size, gives the same sums up to the order of their folds; at the
smallest angle every group opens all leaves and the sums are the exact ones."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _eval(dwglib, h, q, grad):
    w = np.zeros(len(q), np.float32)
    g = np.zeros((len(q), 3), np.float32) if grad else None
    dwglib.dwg_eval_gwn(h, q, w, g)
    return w, g


@pytest.mark.parametrize("n", [1, 17, 300, 5000])
@pytest.mark.parametrize("lam", [0.0, 25.0])
def test_prefix_of_a_call(dwglib, n, lam):
    p, nt = synth.torus(n, seed=n, noise=0.001)
    q = synth.uniform_box(4096 + 65, [-1.5] * 3, [1.5] * 3, seed=2)
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_weights(h, np.full(n, 11.8 / n, np.float32))
        dwglib.dwg_set_params(h, 1 if lam else 0, 0.03, lam, 10, 0.1)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE, 0.5)
        dwglib.dwg_set_normals(h, nt.astype(np.float32))
        wf, gf = _eval(dwglib, h, q, True)
        # FP32 terms, compensated folds: the same terms in other items differ
        # by the rounding of (hi, lo) to float, far inside 1e-6 of the scale
        ws, gs = np.abs(wf).max(), np.abs(gf).max()
        for m in (1, 63, 64, 65, 640):
            k = m // 64 * 64 if m % 64 else m  # whole groups: the same boxes
            w, g = _eval(dwglib, h, np.ascontiguousarray(q[:m]), True)
            assert np.all(np.isfinite(w)) and np.all(np.isfinite(g))
            assert np.abs(w[:k] - wf[:k]).max(initial=0.0) <= 1e-6 * ws
            assert np.abs(g[:k] - gf[:k]).max(initial=0.0) <= 1e-6 * gs
        w1, _ = _eval(dwglib, h, q, False)
        assert np.abs(w1 - wf).max() <= 1e-6 * ws
        # every node open: the exact sums
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE, 1e-4)
        wt, gt = _eval(dwglib, h, q, True)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_ALLPAIRS, 0.5)
        we, ge = _eval(dwglib, h, q, True)
        assert np.abs(wt - we).max() <= 1e-5 * max(1.0, ws)
        assert np.abs(gt - ge).max() <= 1e-5 * max(1.0, np.abs(ge).max())
    finally:
        dwglib.dwg_destroy(h)
