"""Verification batches at the edges of their kernels: the weighted sums of long batches on the tensor
cores give the transcripts of the CUDA-core kernels word for word (block counts around the threshold,
ragged last blocks and tiles), and the layers' batches over GF(2^64) the oracle's at sizes with no, one
and several folding launches and odd dimensions on the way."""
import numpy as np
import pytest

from oracle import nonlinear as NL
from oracle import protocols as OP
from oracle.boolean import BoolSession
from oracle.shares import Session
from paper_2411_09287_gb300 import workloads

from test_gpu_nonlinear import (assert_shared_equal, check_layer_trace, gpu_shared, mpc,  # noqa: F401
                                seed_of, signed)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(1 << 16) - 1, 1 << 16, (1 << 16) + 1, 70001])
def test_long_mult_batch_transcripts(mpc, n):  # noqa: F811
    x, y = (workloads.uniform_words(n, f"long-{n}-{q}") for q in "xy")
    out = []
    for path in (0, 1):
        ctx = mpc.Context(seed_of("long-mult"), gemm_path=path)
        gx, gy = ctx.share_input(1, x), ctx.share_input(2, y)
        gz = ctx.mult(3, gx, gy, n)
        rc, tr = ctx.verify_mult(4, gx, gy, gz, n, 3, trace=True)
        assert rc == mpc.MPC_OK
        out.append((mpc.to_u64(gz), mpc.to_u64(tr)))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n", [1, 960, 1023, 1025, 4096, 4161])
def test_relu_transcripts_of_both_paths(mpc, n):  # noqa: F811
    vals = np.random.default_rng(n).integers(-2 ** 45, 2 ** 45, n).view(np.uint64)
    out = []
    for path in (0, 1):
        ctx = mpc.Context(seed_of("relu-paths"), gemm_path=path)
        rc, res, tr = ctx.relu(2, 3, ctx.share_input(1, vals), n, trace=True)
        assert rc == mpc.MPC_OK
        out.append((mpc.to_u64(res), mpc.to_u64(tr)))
        assert np.array_equal(signed(ctx.reconstruct(res, n)), np.maximum(signed(vals), 0))
    assert np.array_equal(out[0][0], out[1][0])
    assert np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("n", [1, 150, 290])
def test_relu_layer_transcript(mpc, n):  # noqa: F811
    seed = seed_of(f"relu-layer-{n}")
    vals = np.random.default_rng(n).integers(-2 ** 40, 2 ** 40, n).view(np.uint64)
    ctx = mpc.Context(seed)
    s, bs = Session(seed), BoolSession(seed)
    rc, out, tr = ctx.relu(2, 3, ctx.share_input(1, vals), n, trace=True)
    assert rc == mpc.MPC_OK
    oout, triples = NL.relu(s, bs, OP.share_input(s, vals, 1), 2)
    otr = {"mult": [], "inner": [], "and": [], "eda": []}
    assert NL.verify_layer(s, bs, triples, 3, trace=otr)
    assert_shared_equal(gpu_shared(mpc, out, n), oout, "relu out")
    check_layer_trace(mpc, tr, otr, [64 * ((n + 63) // 64)])


@pytest.mark.parametrize("site", ["MZ1", "MZ2", "HIGH_BIT", "REC_MSG"])
def test_relu_rejects_each_message(mpc, site):  # noqa: F811
    vals = np.random.default_rng(7).integers(-2 ** 40, 2 ** 40, 64).view(np.uint64)
    ctx = mpc.Context(seed_of(f"relu-site-{site}"))
    gx = ctx.share_input(1, vals)
    ctx.inject_fault(site, 77, 1 << 9)
    rc, _, _ = ctx.relu(2, 3, gx, 64)
    assert rc in (mpc.MPC_ERR_VERIFY, mpc.MPC_ERR_ABORT)
