"""dwg_mlp_grad over several tiles a CTA against the same rows in parts of one
tile a CTA.  The gradient is that of a mean, so the whole is the mean of equal
parts' gradients; with 2 or 4 parts every factor is a power of two, and the
same bf16 products are summed in another order.  The last rows' targets are
far off, so that the last, short tile weighs as much as a full one.

Sums of up to 40,000 fp32 products in two orders differ by some 1e-6 of the
sum of their magnitudes, about 1e-5 of a matrix's largest entry; a lost tile
of 64 rows is one in 305 to 1,216, over 1e-3 of it at 608."""
import numpy as np
import pytest

import synth
from oracle import mlp

pytestmark = pytest.mark.gpu

ONE_TILE = 2 * 152 * 64  # rows up to which each CTA has one tile


@pytest.mark.parametrize("parts,rows", [(2, 9729), (2, 19455), (4, 9729), (4, 19456)])
def test_whole_and_parts(dwglib, parts, rows):
    torch = pytest.importorskip("torch")
    assert rows <= ONE_TILE
    B = parts * rows
    theta = torch.from_numpy(mlp.init_params(5).astype(np.float32)).cuda()
    X = torch.from_numpy(synth.normal(6, 1, B * 64).reshape(B, 64).astype(np.float32)).cuda()
    T = synth.normal(6, 2, B * 3).reshape(B, 3).astype(np.float32)
    tail = B % 64 or 64
    T[-tail:] *= 64.0 / tail * 4.0
    T = torch.from_numpy(T).cuda()
    g = torch.zeros(mlp.N_PARAMS, device="cuda")

    def run(lo, hi):
        loss = dwglib.dwg_mlp_grad(theta, X[lo:hi].contiguous(), T[lo:hi].contiguous(), g)
        return loss, g.double().cpu().numpy()

    loss, whole = run(0, B)
    got = [run(k * rows, (k + 1) * rows) for k in range(parts)]
    ref = sum(x[1] for x in got) / parts
    assert loss == pytest.approx(sum(x[0] for x in got) / parts, rel=1e-9)
    o = 0
    for name, shape in mlp.SIZES:
        k = int(np.prod(shape))
        err = np.abs(whole[o:o + k] - ref[o:o + k]).max()
        assert err <= 1e-4 * np.abs(ref[o:o + k]).max(), name
        o += k
    # the last tile is seen: without its rows the whole differs by far more
    loss, short = run(0, B - tail)
    w4 = slice(mlp.N_PARAMS - 195, mlp.N_PARAMS - 3)
    lost = 1e-3 * 608 / -(-B // 64)
    assert np.abs(short[w4] * (B - tail) / B - whole[w4]).max() > lost * np.abs(whole[w4]).max()
