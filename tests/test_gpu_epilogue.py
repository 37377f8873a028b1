"""The tensor-core product's protocol epilogue (added masks, a sign, a stream word for every output) on
outputs that fill, miss and exceed a warp's 256 words, with row lengths that are no multiple of a stream
block: every word of the product's sharing equals the u64 path's, with and without truncation."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("t", [-1, 13])
@pytest.mark.parametrize("M,N", [(1, 1), (1, 7), (3, 85), (1, 256), (257, 1), (13, 157), (64, 33), (1025, 3)])
def test_paths_agree(M, N, t):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc, workloads
    K = 5
    X, W = (workloads.uniform_words(n, f"epilogue-{n}") for n in (M * K, K * N))
    out = []
    for path in (0, 1):
        ctx = mpc.Context(hashlib.sha256(b"epilogue").digest(), gemm_path=path)
        zpre, zout, pq = ctx.matmul(3, ctx.share_input(1, X), ctx.share_input(2, W), M, N, K, t)
        ctx.sync()
        out.append([mpc.to_u64(z) for z in (zpre, zout) + ((pq,) if t >= 0 else ())])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
