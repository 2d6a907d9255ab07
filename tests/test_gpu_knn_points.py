"""The points' own nearest neighbours (a shared walk per 32 points, a warp each
for the points it gives up), through the patch features, against dwg_knn's
search of one query per thread in the same (distance, input index) order.
Both subtract in float32, so an entry differs by the scale alone: an RMS of 48
float32 squares, 2^-24 each, and a division: below 4e-6 of the entry."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


def _cloud(kind, n):
    if kind == "copies":   # more copies of a point than the table holds
        return np.ascontiguousarray(np.resize(synth.sphere(max(1, n // 40), seed=3)[0], (n, 3)))
    if kind == "lattice":  # ties at the last neighbour everywhere
        k = int(np.ceil(n ** (1 / 3)))
        g = np.stack(np.meshgrid(*[np.arange(k)] * 3, indexing="ij"), -1).reshape(-1, 3)[:n]
        return np.ascontiguousarray(g / 8.0, dtype=np.float32)
    p = synth.sphere(n, seed=5)[0].copy()
    if kind == "outliers":  # walks that pass the warp's buckets
        p[::7] = 40.0 * synth.normal(9, 1, len(p[::7]) * 3).reshape(-1, 3)
    return np.ascontiguousarray(p, dtype=np.float32)


def _rows(p, at, idx):
    """Offsets of the 16 nearest others of the points `at`, from idx (m, 17)."""
    out = np.zeros((len(at), 48), np.float32)
    for r, i in enumerate(at):
        nb = [j for j in idx[r] if j >= 0 and j != i][:16]
        o = p[nb] - p[i]
        s = np.sqrt((o.astype(np.float64) ** 2).sum(1).mean()) if nb else 0.0
        if s > 0:
            out[r, :3 * len(nb)] = (o / s).ravel()
    return out


def _check(dwglib, p, at, X):
    h = dwglib.dwg_create(p)
    try:
        dwglib.dwg_mlp_features(h, X)
        k = min(17, len(p))
        idx = np.full((len(at), k), -1, np.int64)
        dwglib.dwg_knn(h, np.ascontiguousarray(p[at]), k, idx)
    finally:
        dwglib.dwg_destroy(h)
    got = X[at].cpu().numpy() if hasattr(X, "cpu") else X[at]
    ref = _rows(p, at, idx)
    assert np.all(np.abs(got[:, :48] - ref) <= 4e-6 * np.abs(ref))
    assert np.all(got[:, 51:] == 0) and np.all(np.isfinite(got))


@pytest.mark.parametrize("kind", ["sphere", "lattice", "copies", "outliers"])
@pytest.mark.parametrize("n", [1, 2, 16, 17, 18, 31, 33, 127, 129, 1000, 5003])
def test_points(dwglib, kind, n):
    p = _cloud(kind, n)
    _check(dwglib, p, np.arange(n), np.full((n, 64), 7.0, np.float32))


def test_more_points_than_one_table(dwglib):
    """Past 3 * 2^20 points the table is filled a range at a time: both sides
    of the line (in sorted order, so everywhere in the input)."""
    torch = pytest.importorskip("torch")
    n = (3 << 20) + 33
    p = _cloud("sphere", n)
    X = torch.full((n, 64), 7.0, device="cuda")
    _check(dwglib, p, np.unique(np.concatenate([np.arange(0, n, 1013), np.arange(n - 40, n)])), X)
    assert bool((X != 7.0).all())
