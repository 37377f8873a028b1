"""The im2col rows of narrow kernels (1 to 25 columns), whose blocks take up to 512 rows, against a plain
index map: row counts that fill, miss and exceed whole blocks."""
import hashlib

import numpy as np
import pytest

from test_gpu_im2col import cols_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("geom", [(64, 1, 29, 29, 1, 1, 1, 0), (33, 1, 57, 57, 1, 1, 1, 0),
                                  (40, 2, 28, 31, 1, 1, 1, 0), (17, 1, 60, 60, 2, 2, 2, 1),
                                  (64, 1, 28, 28, 3, 3, 1, 1), (50, 1, 28, 28, 5, 5, 1, 0)])
def test_narrow_rows(geom):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc
    B, C, H, W, kh, kw = geom[:6]
    n = B * C * H * W
    g = np.random.default_rng(6)
    ctx = mpc.Context(hashlib.sha256(b"im2col-narrow").digest())
    xs = ctx.share_input(1, g.integers(0, 1 << 63, n).astype(np.uint64))
    ws = ctx.share_input(2, g.integers(0, 1 << 63, C * kh * kw).astype(np.uint64))
    cols, _, _, _, (M, _, K) = ctx.conv2d(3, xs, ws, geom, 1)
    got = mpc.to_u64(cols)[: 6 * M * K].reshape(6, -1)
    comps = mpc.to_u64(xs)[: 6 * n].reshape(6, -1)
    for c in range(6):
        assert np.array_equal(got[c], cols_of(comps[c], geom))
