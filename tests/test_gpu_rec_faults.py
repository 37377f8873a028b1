"""Pi_Rec's hash comparison at every opening of a verification: a corrupted P0 -> P1 message of the
challenge r, of any round's zeta' (block, dense, short and S-matrix rounds, the AND gates' batch) or of
Delta makes the call abort, whichever opening it hits and however many are recorded before it; past the
last opening the fault does not fire and the call accepts."""
import numpy as np
import pytest

from oracle import protocols as OP
from oracle import verify as OV
from oracle.shares import Session
from paper_2411_09287_gb300 import workloads

from test_gpu_parity import mpc, seed_of  # noqa: F401

pytestmark = pytest.mark.gpu


def _outcomes(mpc, run, openings, **kw):  # noqa: F811
    """run(ctx, arm) for a fault at each opening, and for one past the last."""
    for skip in range(openings + 1):
        ctx = mpc.Context(seed_of("rec-faults"), **kw)
        rc = run(ctx, lambda: ctx.inject_fault("REC_MSG", 21, 1 << 33, skip=skip))
        assert rc == (mpc.MPC_OK if skip == openings else mpc.MPC_ERR_ABORT), skip
        ctx.close()


@pytest.mark.parametrize("n,R,path", [(5, 3, 1), (777, 45, 1), (777, -1, 0), (70001, -1, 1)])
def test_mult_batch_openings(mpc, n, R, path):  # noqa: F811
    x = workloads.uniform_words(n, "rec-faults")

    def run(ctx, arm):
        gx = ctx.share_input(1, x)
        gz = ctx.mult(2, gx, gx, n)
        arm()
        return ctx.verify_mult(3, gx, gx, gz, n, 2, R=R)[0]

    _outcomes(mpc, run, (mpc.default_R(n) if R < 0 else R) + 2, gemm_path=path)


@pytest.mark.parametrize("path", [0, 1])
def test_layer_openings(mpc, path):  # noqa: F811
    M, N, K, t = 12, 20, 130, 13
    X, W = workloads.gemm_shape(M, N, K, "rec-faults")

    def run(ctx, arm):
        gx, gw = ctx.share_input(1, X), ctx.share_input(2, W)
        zpre, _, pq = ctx.matmul(3, gx, gw, M, N, K, t)
        arm()
        return ctx.verify_matmul(4, gx, gw, zpre, pq, M, N, K, t, 3)[0]

    _outcomes(mpc, run, mpc.default_R(K) + mpc.default_R(64 * M * N) + 4, gemm_path=path)


@pytest.mark.parametrize("path", [0, 1])
def test_relu_openings(mpc, path):  # noqa: F811
    x = np.arange(-20, 50, dtype=np.int64).view(np.uint64)
    rounds = sum(mpc.Context.nonlinear_R([128]))

    def run(ctx, arm):
        gx = ctx.share_input(1, x)
        arm()
        return ctx.relu(2, 3, gx, 70)[0]

    _outcomes(mpc, run, 1 + rounds + 8, gemm_path=path)   # Delta of the comparison, four batches


def test_outcomes_are_the_oracles(mpc):  # noqa: F811
    n, R = 9, 4
    x = workloads.uniform_words(n, "rec-faults-oracle")
    for skip in range(R + 3):
        ctx, sess = mpc.Context(seed_of("rec-faults-o")), Session(seed_of("rec-faults-o"))
        gx, ox = ctx.share_input(1, x), OP.share_input(sess, x, 1)
        gz, oz = ctx.mult(2, gx, gx, n), OP.mult(sess, ox, ox, 2)
        ctx.inject_fault("REC_MSG", 7, 1 << 12, skip=skip)
        sess.arm_fault("REC_MSG", 7, 1 << 12, skip=skip)
        rc, _ = ctx.verify_mult(3, gx, gx, gz, n, 2, R=R)
        try:
            want = mpc.MPC_OK if OV.mult_verify(sess, ox, ox, oz, 3, R=R) else mpc.MPC_ERR_VERIFY
        except OP.Abort:
            want = mpc.MPC_ERR_ABORT
        assert rc == want, skip
