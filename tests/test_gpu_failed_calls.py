"""A call that fails part way leaves nothing behind: the next one is neither
refused for the first one's input nor told of its error."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 3000


@pytest.fixture
def scene(dwglib):
    torch = pytest.importorskip("torch")
    p, nt = synth.sphere(N, seed=6)
    h = dwglib.dwg_create(p)
    dwglib.dwg_set_normals(h, nt.astype(np.float32))
    q = torch.from_numpy(np.ascontiguousarray(1.2 * p, dtype=np.float32)).cuda()
    yield torch, h, q
    dwglib.dwg_destroy(h)


@pytest.mark.parametrize("path", ["exact", "tree"])
@pytest.mark.parametrize("host", [False, True])
def test_invalid_queries_then_no_memory(dwglib, scene, path, host):
    """The queries' copy (48,000 bytes, on the host path 36,000 more) fits, the
    sums' array does not: the invalid query has been seen by then."""
    torch, h, q = scene
    dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE if path == "tree" else dwglib.DWG_PATH_ALLPAIRS, 0.5)
    make = (lambda *s: np.zeros(s, np.float32)) if host else (lambda *s: torch.zeros(*s, device="cuda"))
    ref, w, g = make(N), make(N), make(N, 3)
    good = q.cpu().numpy() if host else q
    bad = good.copy() if host else good.clone()
    bad[7, 1] = float("nan")
    dwglib.dwg_eval_gwn(h, good, ref, g)
    dwglib.dwg_set_scratch(h, 90_000, 0)
    with pytest.raises(dwglib.DWGError) as e:
        dwglib.dwg_eval_gwn(h, bad, w, g)
    assert e.value.code == dwglib.DWG_ERR_OOM
    dwglib.dwg_set_scratch(h)
    dwglib.dwg_eval_gwn(h, good, w, g)
    assert (w == ref).all()
    with pytest.raises(dwglib.DWGError) as e:
        dwglib.dwg_eval_gwn(h, bad, w, g)
    assert e.value.code == dwglib.DWG_ERR_NONFINITE
    dwglib.dwg_eval_gwn(h, good, w, g)
    assert (w == ref).all()


def test_knn_without_memory(dwglib, scene):
    torch, h, q = scene
    idx, ref = (torch.full((N, 10), -7, dtype=torch.int64, device="cuda") for _ in range(2))
    dwglib.dwg_knn(h, q, 10, ref)
    dwglib.dwg_set_scratch(h, 1000, 0)
    with pytest.raises(dwglib.DWGError) as e:
        dwglib.dwg_knn(h, q, 10, idx)
    assert e.value.code == dwglib.DWG_ERR_OOM
    dwglib.dwg_set_scratch(h)
    dwglib.dwg_knn(h, q, 10, idx)
    assert torch.equal(idx, ref)
