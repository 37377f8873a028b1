"""The im2col rows of every share component against a plain index map, with and without the kernel's
column table (up to 1024 columns), ragged last row blocks, strides, padding wider than the kernel's
reach and images smaller than it."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def cols_of(x, geom):
    B, C, H, W, kh, kw, s, p = geom
    Ho, Wo = (H + 2 * p - kh) // s + 1, (W + 2 * p - kw) // s + 1
    xp = np.zeros((B, C, H + 2 * p, W + 2 * p), dtype=np.uint64)
    xp[:, :, p:p + H, p:p + W] = x.reshape(B, C, H, W)
    out = np.empty((B, Ho, Wo, C, kh, kw), dtype=np.uint64)
    for i in range(Ho):
        for j in range(Wo):
            out[:, i, j] = xp[:, :, i * s:i * s + kh, j * s:j * s + kw]
    return out.reshape(-1)


@pytest.mark.parametrize("geom", [(1, 1, 5, 5, 3, 3, 1, 0), (2, 113, 4, 4, 3, 3, 1, 1),
                                  (2, 114, 4, 5, 3, 3, 1, 1), (3, 3, 9, 7, 5, 3, 2, 2),
                                  (1, 2, 2, 3, 3, 5, 1, 4), (5, 1, 1, 1, 1, 1, 1, 0)])
def test_im2col_rows(geom):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc
    B, C, H, W, kh, kw = geom[:6]
    n = B * C * H * W
    g = np.random.default_rng(5)
    ctx = mpc.Context(hashlib.sha256(b"im2col").digest())
    xs = ctx.share_input(1, g.integers(0, 1 << 63, n).astype(np.uint64))
    ws = ctx.share_input(2, g.integers(0, 1 << 63, C * kh * kw * 3).astype(np.uint64))
    cols, _, _, _, (M, _, K) = ctx.conv2d(3, xs, ws, geom, 3)
    got = mpc.to_u64(cols)[: 6 * M * K].reshape(6, -1)
    comps = mpc.to_u64(xs)[: 6 * n].reshape(6, -1)
    for c in range(6):
        assert np.array_equal(got[c], cols_of(comps[c], geom))
