"""mpc_launch_count counts the kernels that ran: the calls' launches as the CUDA activity trace sees
them, at sizes on both sides of the launches that are left out (one-block hash trees, products without an
epilogue) and on both GEMM paths.  The trace is taken in a process of its own."""
import json
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CHILD = """
import hashlib, json
import torch
from torch.profiler import ProfilerActivity, profile
from paper_2411_09287_gb300 import mpc

def layer(ctx, M, N, K):
    a = torch.arange(M * K, device="cuda", dtype=torch.int64)
    b = torch.arange(K * N, device="cuda", dtype=torch.int64)
    x, w = ctx.share_input(1, a), ctx.share_input(2, b)
    zpre, zout, pq = ctx.matmul(3, x, w, M, N, K, 13)
    assert ctx.verify_matmul(4, x, w, zpre, pq, M, N, K, 13, 3)[0] == 0
    z = ctx.mult(5, x, x, M * K)
    assert ctx.verify_mult(6, x, x, z, M * K, 5)[0] == 0
    out, tpq = ctx.trunc(7, z, M * K, 5)
    assert ctx.verify_trunc(8, tpq, M * K, 5, 7)[0] == 0
    assert ctx.relu(9, 10, out, M * K)[0] == 0
    ctx.reconstruct(out, M * K, to_host=False)
    ctx.reconstruct_noalloc(out, M * K)

with profile(activities=[ProfilerActivity.CUDA]):   # the first trace of a process can be empty
    torch.zeros(1, device="cuda")
    torch.cuda.synchronize()
res = []
for path in (0, 1):
    for M, N, K in ((3, 5, 7), (96, 40, 100)):
        ctx = mpc.Context(hashlib.sha256(b"launch-count").digest(), gemm_path=path)
        layer(ctx, M, N, K)
        torch.cuda.synchronize()
        n0 = ctx.launch_count()
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            layer(ctx, M, N, K)
            torch.cuda.synchronize()
        names = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA]
        res.append([path, M, ctx.launch_count() - n0, sum("mpc3" in n or "k_" in n for n in names),
                    len(names)])
print("RESULT " + json.dumps(res))
"""


def test_launch_count_matches_the_trace():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    r = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    res = json.loads(next(line for line in r.stdout.splitlines() if line.startswith("RESULT "))[7:])
    if not any(events for *_, events in res):
        pytest.skip("no activity trace on this machine")
    for path, M, counted, traced, _ in res:
        assert counted == traced, (path, M, counted, traced)
