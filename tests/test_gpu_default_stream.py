"""Callers' device arrays with work still pending on the default stream: calls
read them behind what fills them, and write them behind what still reads them,
although a handle's own stream is not ordered with the default stream."""
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 3000


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


@pytest.fixture
def scene(dwglib, torch):
    p, nt = synth.sphere(N, seed=1)
    p = torch.from_numpy(np.ascontiguousarray(p, dtype=np.float32)).cuda()
    nt = torch.from_numpy(nt.astype(np.float32)).cuda()
    h = dwglib.dwg_create(p)
    dwglib.dwg_set_params(h, 0, 0.02, 0.0, 2, 0.1)
    dwglib.dwg_set_update(h, 5, 10, dwglib.DWG_UPDATE_LEVELSET)
    dwglib.dwg_set_normals(h, nt)
    a = torch.ones(4096, 4096, device="cuda")

    def busy():  # tens of milliseconds of work on the default stream
        x = a
        for _ in range(20):
            x = (x @ x) * 1e-4
        return x

    busy()
    torch.cuda.synchronize()
    yield h, p, nt, busy
    dwglib.dwg_destroy(h)


def _net(torch, d):
    P = np.load(os.path.join(os.path.dirname(os.path.abspath(d.__file__)), "warm_start.npy"))
    return torch.from_numpy(P.astype(np.float32)).cuda()


def _normals(d, torch, h):
    o = torch.empty(N, 3, device="cuda")
    d.dwg_get_normals(h, o)
    return o


def _eval(d, torch, h, q):
    w = torch.empty(N, device="cuda")
    d.dwg_eval_gwn(h, q, w)
    return w


def _knn(d, torch, h, q):
    i = torch.empty(N, 5, dtype=torch.int64, device="cuda")
    d.dwg_knn(h, q, 5, i)
    return i


def _created(d, torch, q):
    h2 = d.dwg_create(q)
    try:
        return _knn(d, torch, h2, q)
    finally:
        d.dwg_destroy(h2)


@pytest.mark.parametrize("what", ["queries", "knn", "normals", "weights", "start", "network",
                                  "points"])
def test_inputs(dwglib, torch, scene, what):
    d, (h, p, nt, busy) = dwglib, scene
    final = {"queries": 1.2 * p, "knn": 0.9 * p, "normals": nt.flip(0).contiguous(),
             "weights": torch.rand(N, device="cuda") + 0.5, "start": nt.flip(0).contiguous(),
             "network": _net(torch, d), "points": 2.0 * p}[what].contiguous()
    use = {
        "queries": lambda x: _eval(d, torch, h, x),
        "knn": lambda x: _knn(d, torch, h, x),
        "normals": lambda x: (d.dwg_set_normals(h, x), _normals(d, torch, h))[1],
        "weights": lambda x: (d.dwg_set_weights(h, x), _eval(d, torch, h, 1.2 * p))[1],
        "start": lambda x: (d.dwg_set_init(h, d.DWG_INIT_GIVEN, 1, x), _normals(d, torch, h))[1],
        "network": lambda x: (d.dwg_set_init(h, d.DWG_INIT_LEARNED, 1, x),
                              _normals(d, torch, h))[1],
        "points": lambda x: _created(d, torch, x),
    }[what]
    torch.cuda.synchronize()
    ref = use(final)
    x = torch.ones_like(final)
    use(torch.ones_like(final) * 0.5 if what not in ("points",) else p)  # another call before
    torch.cuda.synchronize()
    busy()
    x.copy_(final)
    got = use(x)
    torch.cuda.synchronize()
    assert torch.equal(got, ref)


@pytest.mark.parametrize("what", ["w", "grad", "idx", "normals", "triangles", "areas", "radii",
                                  "features"])
def test_outputs(dwglib, torch, scene, what):
    d, (h, p, nt, busy) = dwglib, scene
    q = (1.2 * p).contiguous()
    cnt, _ = d.dwg_extract_level_set(h)
    shape = {"w": (N,), "grad": (N, 3), "idx": (N, 5), "normals": (N, 3), "triangles": (cnt, 9),
             "areas": (N,), "radii": (N,), "features": (N, 64)}[what]
    out = torch.full(shape, 7, device="cuda",
                     dtype=torch.int64 if what == "idx" else torch.float32)
    keep = torch.empty_like(out)
    call = {
        "w": lambda: d.dwg_eval_gwn(h, q, out),
        "grad": lambda: d.dwg_eval_gwn(h, q, torch.empty(N, device="cuda"), out),
        "idx": lambda: d.dwg_knn(h, q, 5, out),
        "normals": lambda: d.dwg_get_normals(h, out),
        "triangles": lambda: d.dwg_extract_level_set(h, out),
        "areas": lambda: d.dwg_voronoi_weights(h, 15, out),
        "radii": lambda: d.dwg_set_regularization(h, d.DWG_REG_CLAMP, 10, 0.0, 0.0, out),
        "features": lambda: d.dwg_mlp_features(h, out),
    }[what]
    torch.cuda.synchronize()
    busy()
    keep.copy_(out)  # still pending when the call writes
    call()
    torch.cuda.synchronize()
    assert bool((keep == 7).all()) and not bool((out == 7).all())
