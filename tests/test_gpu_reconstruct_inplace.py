"""Pi_Rec whose output lies in the sharing it opens: each component in turn, and across components 0 and
1, opens the right words and passes the hash comparison (the hashed components are read before the
opening overwrites them), with a caller's workspace and with the library's own array."""
import hashlib

import ctypes as C
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 300, 70001])
@pytest.mark.parametrize("at", [0, 0.5, 1, 2, 3, 4, 5])
def test_output_inside_the_sharing(n, at):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc, workloads
    x = workloads.uniform_words(n, f"inplace-{n}")
    ctx = mpc.Context(hashlib.sha256(b"inplace").digest())
    gx = ctx.share_input(1, x)
    off = int(at * n)
    for noalloc in (False, True):
        s = gx.clone()
        out = C.c_void_p(s.data_ptr() + 8 * off)
        if noalloc:
            rc = ctx.lib.mpc_reconstruct_noalloc(ctx.h, C.c_void_p(s.data_ptr()), n, out)
        else:
            wsb = ctx.ws_size(mpc.OP_RECONSTRUCT, n)
            ws = ctx.workspace(wsb)
            rc = ctx.lib.mpc_reconstruct(ctx.h, C.c_void_p(s.data_ptr()), n, out, 0,
                                         C.c_void_p(ws.data_ptr()), wsb)
        assert rc == mpc.MPC_OK
        assert np.array_equal(mpc.to_u64(s)[off:off + n], x)
