"""Clouds at the lines below which a call takes fewer launches: neighbours
searched by the kernel that uses them (48 points), the centroid (512) and the
mean area (2,048) summed by one block."""
import numpy as np
import pytest

import synth
from test_gpu_knn_points import _check, _cloud

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["sphere", "lattice", "copies"])
@pytest.mark.parametrize("n", [47, 48, 49])
def test_neighbours(dwglib, kind, n):
    _check(dwglib, _cloud(kind, n), np.arange(n), np.full((n, 64), 7.0, np.float32))


@pytest.mark.parametrize("n", [1, 511, 512, 513, 1025])
def test_centroid(dwglib, n):
    """Columns 48 to 50 are (p - c) / R in FP64, rounded to float32 once."""
    p = np.ascontiguousarray(synth.torus(n, seed=n, noise=0.01)[0] + 5.0, dtype=np.float32)
    h = dwglib.dwg_create(p)
    try:
        X = np.full((n, 64), 7.0, np.float32)
        dwglib.dwg_mlp_features(h, X)
    finally:
        dwglib.dwg_destroy(h)
    q = p.astype(np.float64)
    q -= q.mean(0)
    R = np.sqrt((q * q).sum(1).mean())
    ref = q / R if R > 0 else q
    # 2^-24 of the entry, and the centroid to 2^-53 of the coordinates' size
    assert np.all(np.abs(X[:, 48:51] - ref) <= 6.1e-8 * np.abs(ref) + 1e-14)


@pytest.mark.parametrize("n", [2047, 2048, 2049])
def test_mean_area(dwglib, n):
    """A point whose neighbourhood has no extent (copies of one point) takes the
    mean of the positive areas."""
    p = np.ascontiguousarray(synth.sphere(n, seed=9)[0], dtype=np.float32)
    p[:40] = [3.0, 0.0, 0.0]
    a = np.zeros(n, np.float32)
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_voronoi_weights(h, 15, a)
    finally:
        dwglib.dwg_destroy(h)
    mean = a[40:].astype(np.float64).mean()
    assert np.all(a[:40] == a[0]) and abs(a[0] / mean - 1.0) <= 1e-6
