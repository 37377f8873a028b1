"""Pi_MultVerify^R against the oracle at the edges of its round structure: batches of one element
to several blocks, odd sizes, R from none to more rounds than the batch has bits (and more opened
challenges than one hash launch records), both readings of the third interpolation point and both
GEMM paths.  Every revealed challenge, every share of h(0) and h(p2) and the opened Delta agree."""
import numpy as np
import pytest

from oracle import protocols as OP
from oracle import verify as OV
from oracle.shares import Session
from paper_2411_09287_gb300 import workloads

from test_gpu_parity import assert_ledger, check_trace, mpc, seed_of  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("mode,path", [(0, 1), (1, 1), (0, 0)])
@pytest.mark.parametrize("n,R", [(1, 0), (1, 2), (2, 1), (7, 3), (8, 3), (9, 4), (15, 1), (17, 2),
                                 (63, 6), (65, 5), (130, 0), (513, 4), (777, 45), (1100, -1)])
def test_mult_verify_rounds(mpc, n, R, mode, path):  # noqa: F811
    seed = seed_of(f"rounds-{n}-{R}")
    x, y = (workloads.uniform_words(n, f"rounds-{n}-{q}") for q in "xy")
    ctx = mpc.Context(seed, reduce_mode=mode, gemm_path=path)
    sess = Session(seed, reduce_mode="x" if mode == 0 else "zeta2")
    gx, gy = ctx.share_input(1, x), ctx.share_input(2, y)
    gz = ctx.mult(3, gx, gy, n)
    ox, oy = OP.share_input(sess, x, 1), OP.share_input(sess, y, 2)
    oz = OP.mult(sess, ox, oy, 3)
    rc, tr = ctx.verify_mult(4, gx, gy, gz, n, 3, R=R, trace=True)
    otr = []
    ok = OV.mult_verify(sess, ox, oy, oz, 4, R=None if R < 0 else R, trace=otr)
    assert ok and rc == mpc.MPC_OK
    check_trace(mpc, tr, otr, [mpc.default_R(n) if R < 0 else R])
    assert_ledger(mpc, ctx, sess)
    assert np.array_equal(ctx.reconstruct(gz, n), x * y)
