"""Calls beside a capture on a stream that is ordered with the default stream
(made without cudaStreamNonBlocking): nothing may be queued on the default
stream then, so the call neither breaks the capture nor reads its arrays before
what the default stream already held."""
import ctypes
import threading

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


@pytest.fixture
def blocking(torch):
    rt = torch.cuda.cudart()
    torch.cuda.current_stream()
    raw = ctypes.c_void_p()
    assert int(rt.cudaStreamCreate(ctypes.addressof(raw))) == 0
    yield torch.cuda.ExternalStream(raw.value)
    torch.cuda.synchronize()
    rt.cudaStreamDestroy(raw.value)


@pytest.mark.parametrize("mode", ["thread_local", "relaxed"])
@pytest.mark.parametrize("path", ["exact", "tree"])
def test_eval_beside_a_capture_ordered_with_the_default_stream(dwglib, torch, blocking, mode, path):
    n = 3000
    p, nrm = synth.sphere(n, seed=1)[:2]
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE if path == "tree"
                            else dwglib.DWG_PATH_ALLPAIRS, 0.5)
        dwglib.dwg_set_normals(h, np.ascontiguousarray(nrm, dtype=np.float32))
        q0 = torch.from_numpy(np.ascontiguousarray(1.3 * p, dtype=np.float32)).cuda()
        ref, w = torch.empty(n, device="cuda"), torch.empty(n, device="cuda")
        for _ in range(2):
            dwglib.dwg_eval_gwn(h, q0, ref)
        q, y = torch.zeros_like(q0), torch.zeros(10, device="cuda")
        a = torch.ones(4096, 4096, device="cuda")
        torch.cuda.synchronize()
        for _ in range(20):  # tens of milliseconds in front of the queries
            a = (a @ a) * 1e-4
        q.copy_(q0)
        seen = []

        def call():
            try:
                dwglib.dwg_eval_gwn(h, q, w)
            except Exception as e:
                seen.append(e)

        g = torch.cuda.CUDAGraph()
        with torch.cuda.stream(blocking):
            g.capture_begin(capture_error_mode=mode)
            y.add_(1)
            t = threading.Thread(target=call)
            t.start()
            t.join()
            y.add_(1)
            g.capture_end()
        torch.cuda.synchronize()
        g.replay()
        torch.cuda.synchronize()
        assert not seen and float(y[0]) == 2.0 and torch.equal(w, ref)
    finally:
        dwglib.dwg_destroy(h)
