"""The scratch of a handle's calls, handed out in pieces of kept segments: calls
of many kinds and sizes one after the other on a handle that keeps it give the
bits of the same calls on a handle that keeps none, with the default bound, a
small one and none in turn."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 6000


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


def _handle(d):
    p, nt = synth.torus(N, seed=3, noise=0.002)
    h = d.dwg_create(np.ascontiguousarray(p, dtype=np.float32))
    d.dwg_set_params(h, 1, 0.03, 10.0, 2, 0.1)
    d.dwg_set_update(h, 6, 10, d.DWG_UPDATE_LEVELSET)
    d.dwg_set_normals(h, nt.astype(np.float32))
    return h


def _call(d, torch, h, q, kind, m, host):
    new = (lambda *s: np.full(s, 7.0, np.float32)) if host else \
        (lambda *s: torch.full(s, 7.0, device="cuda"))
    x = q[:m].cpu().numpy() if host else q[:m].contiguous()
    if kind in ("exact", "tree"):
        d.dwg_set_tree(h, d.DWG_PATH_TREE if kind == "tree" else d.DWG_PATH_ALLPAIRS, 0.5)
        out = [new(m), new(m, 3)]
        d.dwg_eval_gwn(h, x, *out)
    elif kind == "knn":
        idx = np.full((m, 12), -7, np.int64)
        out = [idx if host else torch.from_numpy(idx).cuda()]
        d.dwg_knn(h, x, 12, out[0])
    elif kind == "features":
        out = [new(N, 64)]
        d.dwg_mlp_features(h, out[0])
    elif kind == "weights":
        out = [new(N)]
        d.dwg_voronoi_weights(h, 15, out[0])
    else:
        d.dwg_set_tree(h, d.DWG_PATH_ALLPAIRS, 0.5)
        n0 = new(N, 3)
        d.dwg_get_normals(h, n0)
        cnt, iso = d.dwg_extract_level_set(h)
        out = [n0, np.array([cnt, iso])]
    return [o if isinstance(o, np.ndarray) else o.cpu().numpy() for o in out]


def test_mixed_calls(dwglib, torch):
    d = dwglib
    rng = np.random.default_rng(4)
    q = torch.from_numpy(synth.uniform_box(40000, [-1.5] * 3, [1.5] * 3, seed=2)
                         .astype(np.float32)).cuda()
    kept, none = _handle(d), _handle(d)
    try:
        d.dwg_set_scratch(none, -1, 0)
        for i in range(90):
            if i % 30 == 20:
                d.dwg_set_scratch(kept, -1, int(rng.integers(0, 3 << 20)))
            elif i % 30 == 0:
                d.dwg_set_scratch(kept)
            kind = ["exact", "tree", "knn", "features", "weights", "level set"][rng.integers(6)]
            m = int(np.exp(rng.uniform(0, np.log(40000))))
            host = bool(rng.integers(2))
            a = _call(d, torch, kept, q, kind, m, host)
            b = _call(d, torch, none, q, kind, m, host)
            for x, y in zip(a, b):
                assert np.array_equal(x, y), (i, kind, m)
    finally:
        d.dwg_destroy(kept)
        d.dwg_destroy(none)
