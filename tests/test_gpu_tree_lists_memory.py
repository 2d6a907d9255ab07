"""A Barnes-Hut call whose lists do not fit into its scratch walks the tree
instead of failing: the same terms per query either way, so the same sums up to the order of their folds (FP32 terms,
compensated folds: far inside 1e-6 of the scale, as for work items of another
size).  Also more queries than one range of groups holds."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N, M = 20000, 20000
RANGE = 16384 * 64  # queries of one range of groups


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


def _handle(dwglib, n, lam):
    p, nt = synth.torus(n, seed=n, noise=0.001)
    h = dwglib.dwg_create(p)
    dwglib.dwg_set_weights(h, np.full(n, 11.8 / n, np.float32))
    dwglib.dwg_set_params(h, 1 if lam else 0, 0.03, lam, 10, 0.1)
    dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE, 0.5)
    dwglib.dwg_set_normals(h, nt.astype(np.float32))
    return h


def _queries(torch, m):
    q = synth.uniform_box(m, [-1.5] * 3, [1.5] * 3, seed=2)  # in no order: long lists
    return torch.from_numpy(np.ascontiguousarray(q, dtype=np.float32)).cuda()


def _eval(dwglib, torch, h, q, grad=True):
    w = torch.full((len(q),), float("nan"), device="cuda")
    g = torch.full((len(q), 3), float("nan"), device="cuda") if grad else None
    dwglib.dwg_eval_gwn(h, q, w, g)
    return [w, g] if grad else [w]


def _same(a, b):
    for x, y in zip(a, b):
        assert bool(x.isfinite().all())
        assert float((x - y).abs().max()) <= 1e-6 * float(y.abs().max())


@pytest.mark.parametrize("lam", [0.0, 25.0])
@pytest.mark.parametrize("limit", [5 << 20, 980_000, 965_000])
def test_less_scratch_than_the_lists(dwglib, torch, limit, lam):
    """The call's own arrays (queries 320,000 bytes, partial sums 640,000,
    offsets 13 KB) leave room for blocks smaller than the lists, and at 980,000
    bytes for the arrays alone, at 965,000 not for the offsets."""
    h = _handle(dwglib, N, lam)
    try:
        q = _queries(torch, M)
        ref = _eval(dwglib, torch, h, q)
        records = dwglib.dwg_get_stats(h)["interactions_eval"] / 64
        # an item holds at most 2,048 records and writes 2,048 bytes: no block
        # of this limit holds the call's items, let alone its lists
        assert records > limit
        dwglib.dwg_set_scratch(h, limit, -1)
        _same(_eval(dwglib, torch, h, q), ref)
        assert dwglib.dwg_get_stats(h)["interactions_eval"] / 64 == records
        _same(_eval(dwglib, torch, h, q, False), ref)
        dwglib.dwg_set_scratch(h, -1, 0)
        _same(_eval(dwglib, torch, h, q), ref)
    finally:
        dwglib.dwg_destroy(h)


def test_too_little_for_the_call_itself(dwglib, torch):
    h = _handle(dwglib, N, 0.0)
    try:
        q = _queries(torch, M)
        ref = _eval(dwglib, torch, h, q)
        dwglib.dwg_set_scratch(h, 400_000, 0)
        with pytest.raises(dwglib.DWGError) as e:
            _eval(dwglib, torch, h, q)
        assert e.value.code == dwglib.DWG_ERR_OOM
        dwglib.dwg_set_scratch(h)
        _same(_eval(dwglib, torch, h, q), ref)
        with pytest.raises(dwglib.DWGError) as e:
            dwglib.dwg_set_scratch(h, -2, 0)
        assert e.value.code == dwglib.DWG_ERR_INVALID
    finally:
        dwglib.dwg_destroy(h)


@pytest.mark.parametrize("limit", [-1, 64 << 20])
def test_more_queries_than_one_range(dwglib, torch, limit):
    """Both sides of the line, and a last group that is not full; with a limit
    that the first range's lists do not fit into and the second's do."""
    h = _handle(dwglib, 300, 25.0)
    try:
        q = _queries(torch, RANGE + 130)
        dwglib.dwg_set_scratch(h, limit, -1)
        w, g = _eval(dwglib, torch, h, q)
        for a, b in ((0, 640), (RANGE - 640, RANGE), (RANGE, RANGE + 130)):
            _same([w[a:b], g[a:b]], _eval(dwglib, torch, h, q[a:b].contiguous()))
    finally:
        dwglib.dwg_destroy(h)


@pytest.mark.parametrize("m", [RANGE + 130, 2 * RANGE + 130])
def test_more_lists_than_a_call_makes(dwglib, torch, m):
    """300,000 sources, queries in no order: every group opens most leaves, over
    18,000 entries a group, 300M in a full range -- more than 1 GB, so one or
    two ranges are walked; the last range's lists fit."""
    h = _handle(dwglib, 300_000, 25.0)
    try:
        q = _queries(torch, m)
        w, g = _eval(dwglib, torch, h, q)
        for a, b in ((0, 640), (RANGE - 640, RANGE), (RANGE, RANGE + 128), (m - 130, m)):
            _same([w[a:b], g[a:b]], _eval(dwglib, torch, h, q[a:b].contiguous()))
    finally:
        dwglib.dwg_destroy(h)
