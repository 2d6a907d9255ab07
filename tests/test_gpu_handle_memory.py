"""Device memory of handles: what a handle took is free again once it is
destroyed, whichever path it ran."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


def _free(torch):
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def _once(dwglib, p, out, what):
    if what == "batch":
        h = dwglib.dwg_create_batch(p, [0, 9000, len(p)])
    else:
        h = dwglib.dwg_create(p)
        dwglib.dwg_set_update(h, 8, 10, dwglib.DWG_UPDATE_LEVELSET)
        dwglib.dwg_set_tree(h, dwglib.DWG_PATH_TREE if what == "tree"
                            else dwglib.DWG_PATH_ALLPAIRS, 0.5)
    try:
        dwglib.dwg_set_params(h, 0, 0.01, 0.0, 2, 0.1)
        if what == "batch":
            dwglib.dwg_orient_batch(h, out, 2)
        elif what == "level set":
            dwglib.dwg_extract_level_set(h)
        else:
            dwglib.dwg_orient(h, out)
    finally:
        dwglib.dwg_destroy(h)


@pytest.mark.parametrize("what", ["exact", "tree", "level set", "batch"])
def test_destroy_gives_everything_back(dwglib, torch, what):
    """The lattice of a 40,000-point cloud at depth 8 alone is over 4 MB, so 12
    handles that kept it would hold 48 MB; the driver hands memory out in
    blocks of 2 MB, of which a few may stay."""
    p = torch.from_numpy(np.ascontiguousarray(synth.sphere(40000, seed=2)[0])).cuda()
    out = torch.empty_like(p)
    for _ in range(3):
        _once(dwglib, p, out, what)
    before = _free(torch)
    for _ in range(12):
        _once(dwglib, p, out, what)
    assert before - _free(torch) <= 8 * MB


def test_clouds_of_a_batch_keep_as_much_as_one_handle(dwglib, torch):
    """48 clouds of 20,000 points: the scratch that their Voronoi weights and
    their octrees took, some 14 MB a cloud, is not kept 48 times over."""
    k, n = 48, 20000
    p = torch.from_numpy(np.ascontiguousarray(synth.sphere(n, seed=2)[0])).cuda()
    p = (p[None] + 3.0 * torch.arange(k, device="cuda")[:, None, None]).reshape(-1, 3).contiguous()
    out = torch.empty_like(p)
    h = dwglib.dwg_create_batch(p, np.arange(k + 1, dtype=np.int64) * n)
    try:
        for build in (lambda: dwglib.dwg_voronoi_weights(h, 15),
                      lambda: dwglib.dwg_orient_batch(h, out, k)):
            dwglib.dwg_set_params(h, 0, 0.0, 0.0, 1, 0.1)
            dwglib.dwg_set_scratch(h)
            build()
            held = _free(torch)
            dwglib.dwg_set_scratch(h, -1, 0)
            assert _free(torch) - held <= 300 * MB
        assert _free(torch) - held <= 64 * MB  # what a build took and no call needs
    finally:
        dwglib.dwg_destroy(h)
