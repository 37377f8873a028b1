"""Pi_InnerVerify on long claims (few rounds asked for), a warp a row, against the oracle: at the edge of
its range and past whole blocks of rows, with all components present and with the truncation pairs' two a
side."""
import pytest

from oracle import protocols as OP
from oracle import verify as OV
from oracle.shares import Session
from paper_2411_09287_gb300 import workloads

from test_gpu_parity import check_trace, mpc, seed_of  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,R,path", [(2047, 0, 1), (2048, 0, 1), (2049, 0, 0), (6205, 1, 1)])
def test_mult_batch(mpc, n, R, path):  # noqa: F811
    seed = seed_of(f"long-claim-{n}")
    x, y = (workloads.uniform_words(n, f"long-claim-{n}-{q}") for q in "xy")
    ctx, sess = mpc.Context(seed, gemm_path=path), Session(seed)
    gx, gy = ctx.share_input(1, x), ctx.share_input(2, y)
    gz = ctx.mult(3, gx, gy, n)
    ox, oy = OP.share_input(sess, x, 1), OP.share_input(sess, y, 2)
    oz = OP.mult(sess, ox, oy, 3)
    rc, tr = ctx.verify_mult(4, gx, gy, gz, n, 3, R=R, trace=True)
    otr = []
    assert OV.mult_verify(sess, ox, oy, oz, 4, R=R, trace=otr) and rc == mpc.MPC_OK
    check_trace(mpc, tr, otr, [R])


@pytest.mark.parametrize("fault", [False, True])
def test_layer_with_two_components_a_side(mpc, fault):  # noqa: F811
    M, N, K, t, R = 13, 20, 6, 13, 3   # 64 * 260 / 8 = 2080 elements left
    seed = seed_of("long-claim-layer")
    X, W = workloads.gemm_shape(M, N, K, "long-claim")
    ctx, sess = mpc.Context(seed), Session(seed)
    gx, gw = ctx.share_input(1, X), ctx.share_input(2, W)
    if fault:   # the last output's truncation pair
        ctx.inject_fault("GAMMA2", M * N - 1, 1 << 7)
        sess.arm_fault("GAMMA2", M * N - 1, 1 << 7)
    zpre, _, pq = ctx.matmul(3, gx, gw, M, N, K, t)
    ox, ow = OP.share_input(sess, X, 1), OP.share_input(sess, W, 2)
    res = OP.matmul(sess, ox, ow, 3, trunc_bits=t)
    rc, tr = ctx.verify_matmul(4, gx, gw, zpre, pq, M, N, K, t, 3, -1, R, trace=True)
    otr = []
    ok = OV.matmul_verify(sess, ox, ow, res, 4, t, None, R, trace=otr)
    assert ok == (not fault) and rc == (mpc.MPC_ERR_VERIFY if fault else mpc.MPC_OK)
    check_trace(mpc, tr, otr, [mpc.default_R(K), R])
