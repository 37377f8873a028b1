"""Workspace plans: scratch that lies under buffers of a later step is reserved at its own size, and no
call writes past the bytes that mpc_workspace_size gave for it."""
import hashlib
import os
import re

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
GUARD = 1 << 15      # words after the workspace
PATTERN = 0x5A5A_A5A5_1234_4321


def test_block_batch_reserves_its_digit_planes():
    src = open(os.path.join(ROOT, "paper_2411_09287_gb300", "csrc", "api.cu")).read()
    body = re.search(r"BlkPlan plan_blk\(.*?\n}\n", src, flags=re.S).group(0)
    assert "blk_sums_tc_bytes(" in body


def test_message_buffers_of_a_product():
    """A product plans its messages (three, and four of the truncation pairs) and one copy a fault site,
    not a received copy of every message; a standalone truncation likewise."""
    import ctypes as C

    from paper_2411_09287_gb300 import build
    if not os.path.exists(build.LIB):
        try:
            build.build()
        except RuntimeError as e:      # no toolkit on this host
            pytest.skip(str(e))
    lib = C.CDLL(build.LIB)
    size = lib.mpc_workspace_size
    size.restype = C.c_int64
    size.argtypes = [C.c_void_p, C.c_int] + [C.c_int64] * 3 + [C.c_int] * 3
    OP_MATMUL, OP_TRUNC = 2, 11
    E = 300 * 700
    assert size(None, OP_MATMUL, 300, 700, 50, 13, -1, -1) <= 8 * E * (3 + 4 + 3) + 10 * 256
    assert size(None, OP_MATMUL, 300, 700, 50, -1, -1, -1) <= 8 * E * (3 + 3) + 6 * 256
    assert size(None, OP_TRUNC, E, 0, 0, -1, -1, -1) <= 8 * E * (6 + 4 + 4 + 4) + E   # and the hash trees


@pytest.fixture(scope="module")
def mpc():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc as M
    return M


def _guarded(mpc, monkeypatch, **kw):
    """A context whose every workspace is exactly as large as asked for, followed by guard words."""
    ctx = mpc.Context(hashlib.sha256(b"workspace-plans").digest(), **kw)
    torch, seen = ctx.torch, []

    def workspace(nbytes):
        words = (int(nbytes) + 7) // 8
        t = torch.empty(words + GUARD, dtype=torch.int64, device=ctx.device)
        t[words:] = PATTERN
        seen.append((t, words))
        return t

    monkeypatch.setattr(ctx, "workspace", workspace)
    return ctx, seen


def _untouched(ctx, seen):
    ctx.sync()
    for t, words in seen:
        assert bool((t[words:] == PATTERN).all())


@pytest.mark.gpu
@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("n,R", [(1000, -1), (65535, 4), (65536, 4), (65537, -1), (70001, 5)])
def test_mult_batches_stay_inside(mpc, monkeypatch, path, n, R):
    ctx, seen = _guarded(mpc, monkeypatch, gemm_path=path)
    x = ctx.torch.arange(n, device=ctx.device, dtype=ctx.torch.int64)
    gx = ctx.share_input(1, x)
    gz = ctx.mult(2, gx, gx, n)
    rc, _ = ctx.verify_mult(3, gx, gx, gz, n, 2, R=R)
    assert rc == mpc.MPC_OK
    _untouched(ctx, seen)


@pytest.mark.gpu
@pytest.mark.parametrize("path", [0, 1])
@pytest.mark.parametrize("n", [1, 1024, 4097])
def test_layers_stay_inside(mpc, monkeypatch, path, n):
    ctx, seen = _guarded(mpc, monkeypatch, gemm_path=path)
    x = ctx.torch.arange(-(n // 2), n - n // 2, device=ctx.device, dtype=ctx.torch.int64)
    rc, _, _ = ctx.relu(2, 3, ctx.share_input(1, x), n)
    assert rc == mpc.MPC_OK
    _untouched(ctx, seen)
