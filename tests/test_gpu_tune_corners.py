"""dwg_autotune compares the tree with the evaluator that the exact path runs:
the corners' time of a cloud whose path is left open (and resolves to the tree
before tuning) is that of the same cloud on the exact path.  The general
evaluator that was timed instead takes 1.36 times as long; a repeated timing
differs by some percent."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def test_corner_time_of_an_open_path(dwglib):
    n = 70_000  # above the 65,536 points from which an open path means the tree
    p = np.ascontiguousarray(synth.sphere(n, seed=3)[0], dtype=np.float32)
    ms = []
    for path in (dwglib.DWG_PATH_AUTO, dwglib.DWG_PATH_ALLPAIRS):
        h = dwglib.dwg_create(p)
        try:
            dwglib.dwg_set_params(h, 0, 0.002, 0.0, 2, 0.1)
            dwglib.dwg_set_tree(h, path, 0.5)
            t = dwglib.dwg_autotune(h, dwglib.DWG_TUNE_SHAPES, 1e-3, None)
            assert t["path"] == dwglib.DWG_PATH_ALLPAIRS
            ms.append(t["ms_corners"])
        finally:
            dwglib.dwg_destroy(h)
    assert abs(ms[0] / ms[1] - 1.0) <= 0.15, ms
