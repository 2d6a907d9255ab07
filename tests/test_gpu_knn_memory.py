"""The points' own nearest neighbours with little device scratch: their table is
filled in smaller ranges, with the same bits; where not even the smallest fits
the call returns DWG_ERR_OOM, and the next one with room succeeds."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

N = 20000  # tables of 11 to 18 entries a point: 0.88 to 1.44 MB; the smallest 0.2 to 0.3


@pytest.fixture
def torch():
    return pytest.importorskip("torch")


def _features(d, h, torch):
    X = torch.full((N, 64), 7.0, device="cuda")
    d.dwg_mlp_features(h, X)
    return X


def _voronoi(d, h, torch):
    a = np.zeros(N, np.float32)
    d.dwg_voronoi_weights(h, 15, a)
    return torch.from_numpy(a)


def _pca(d, h, torch):
    o = torch.full((N, 3), 7.0, device="cuda")
    d.dwg_set_init(h, d.DWG_INIT_PCA, 1)
    d.dwg_get_normals(h, o)
    return o


def _radii(d, h, torch):
    r = np.zeros(N, np.float32)
    d.dwg_set_regularization(h, d.DWG_REG_CLAMP, 10, 0.0, 0.0, r)
    return torch.from_numpy(r)


@pytest.mark.parametrize("call", [_features, _voronoi, _pca, _radii])
def test_little_scratch(dwglib, torch, call):
    p = np.ascontiguousarray(synth.sphere(N, seed=5)[0], dtype=np.float32)
    h = dwglib.dwg_create(p)
    try:
        ref = call(dwglib, h, torch)
        # beside the table: up to 170 KB of areas, 80 KB of output
        dwglib.dwg_set_scratch(h, 750_000, 0)
        assert torch.equal(call(dwglib, h, torch), ref)
        dwglib.dwg_set_scratch(h, 100_000, 0)
        with pytest.raises(dwglib.DWGError) as e:
            call(dwglib, h, torch)
        assert e.value.code == dwglib.DWG_ERR_OOM
        dwglib.dwg_set_scratch(h)
        assert torch.equal(call(dwglib, h, torch), ref)
    finally:
        dwglib.dwg_destroy(h)
