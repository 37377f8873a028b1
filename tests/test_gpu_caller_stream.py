"""Verifications on a caller's stream: the batches that leave it for the context's side streams start after
the caller's work enqueued before the call (inputs that arrive late), and the stream covers them when the
call returns (inputs and workspace overwritten at once, the trace read by the next work)."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SLEEP = 40_000_000      # clock cycles, about 20 ms


@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("kind", ["layer", "relu", "pool"])
def test_late_inputs_and_early_reuse(kind, path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc, workloads
    seed = hashlib.sha256(b"caller-stream").digest()
    M, N, K, t = 20, 12, 33, 13
    X, W = workloads.gemm_shape(M, N, K, "caller-stream")
    n = 16 * 12
    vals = workloads.uniform_words(n, "caller-stream") >> np.uint64(2)

    def inputs(ctx):
        if kind != "layer":
            return [ctx.share_input(1, vals)]
        gx, gw = ctx.share_input(1, X), ctx.share_input(2, W)
        zpre, _, pq = ctx.matmul(3, gx, gw, M, N, K, t)
        return [gx, gw, zpre, pq]

    def call(ctx, b):
        if kind == "layer":
            rc, tr = ctx.verify_matmul(4, b[0], b[1], b[2], b[3], M, N, K, t, 3, trace=True)
            return rc, [tr]
        if kind == "relu":
            rc, out, tr = ctx.relu(5, 6, b[0], n, trace=True)
        else:
            rc, out, tr = ctx.maxpool2(5, 6, b[0], (2, 6, 4, 4), trace=True)
        return rc, [out, tr]

    ref = mpc.Context(seed, gemm_path=path)
    rc, want = call(ref, inputs(ref))
    assert rc == mpc.MPC_OK
    torch.cuda.synchronize()

    ctx = mpc.Context(seed, gemm_path=path)
    ready = inputs(ctx)
    torch.cuda.synchronize()
    s = torch.cuda.Stream()
    ctx.set_stream(s)
    with torch.cuda.stream(s):
        for _ in range(2):
            late = [torch.full_like(b, 0x1234567) for b in ready]
            torch.cuda._sleep(SLEEP)
            for a, b in zip(late, ready):
                a.copy_(b)
            rc, got = call(ctx, late)
            for a in late:
                a.zero_()
            ctx._ws.fill_(-1)
            got = [g.clone() for g in got]
            assert rc == mpc.MPC_OK
            s.synchronize()
            for a, b in zip(got, want):
                assert torch.equal(a, b)
