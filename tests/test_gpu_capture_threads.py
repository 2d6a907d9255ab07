"""Calls on one thread while another captures a graph: a caller's own capture
(a torch graph), and the library's capture of its loop on another handle.  The
calls run, the captures hold, the results are those of an undisturbed call."""
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def scene(dwglib):
    torch = pytest.importorskip("torch")
    p, nrm = synth.sphere(4000, seed=1)[:2]
    h = dwglib.dwg_create(p)
    dwglib.dwg_set_normals(h, np.ascontiguousarray(nrm, dtype=np.float32))
    q = torch.from_numpy(np.ascontiguousarray(1.3 * p[:3000])).cuda()
    w = torch.empty(3000, device="cuda")
    dwglib.dwg_eval_gwn(h, q, w)
    torch.cuda.synchronize()
    yield torch, p, h, q, w, w.clone()
    dwglib.dwg_destroy(h)


@pytest.mark.parametrize("mode", ["relaxed", "thread_local"])
def test_eval_beside_a_callers_capture(dwglib, scene, mode):
    torch, p, h, q, w, ref = scene
    x, y = torch.ones(100, device="cuda"), torch.zeros(100, device="cuda")
    torch.cuda.synchronize()
    seen = []

    def call():
        try:
            dwglib.dwg_eval_gwn(h, q, w)
        except Exception as e:
            seen.append(e)

    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, capture_error_mode=mode):
        y.copy_(x * 3)
        t = threading.Thread(target=call)
        t.start()
        t.join()
        y.add_(1)
    g.replay()
    torch.cuda.synchronize()
    assert not seen and float(y[0]) == 4.0 and torch.equal(w, ref)


def test_eval_beside_another_handles_loop(dwglib, scene):
    torch, p, h, q, w, ref = scene
    seen, stop = [], threading.Event()

    def orient():
        h2 = dwglib.dwg_create(np.ascontiguousarray(p[:1500]))
        try:
            out = torch.empty(1500, 3, device="cuda")
            for i in range(20):  # another depth: another graph
                dwglib.dwg_set_update(h2, 4 + (i & 1), 10, dwglib.DWG_UPDATE_LEVELSET)
                dwglib.dwg_orient(h2, out)
        except Exception as e:
            seen.append(e)
        finally:
            dwglib.dwg_destroy(h2)
            stop.set()

    t = threading.Thread(target=orient)
    t.start()
    try:
        while not stop.is_set():
            dwglib.dwg_eval_gwn(h, q, w)
    finally:
        t.join()
    torch.cuda.synchronize()
    assert not seen and torch.equal(w, ref)
