"""The two forms of the S matrix's combination over its blocks, sum_(e_hi) r^(2 L e_hi) S_hi: a product on
the tensor cores from tuning.tc_combine_min blocks on, one pass on the CUDA cores below and on the u64
path.  Both give the same transcript for 2, 3 and 17 blocks (ragged last block included), and the tuning
chooses between them (counted in GR-product launches)."""
import hashlib

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,blocks", [(256, 2), (300, 3), (2177, 18)])
def test_forms_agree_and_tuning_chooses(n, blocks):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2411_09287_gb300 import mpc, workloads
    x = workloads.uniform_words(n, f"combine-{n}")
    out, products = {}, {}
    for name, path, tune in (("default", 1, {}), ("at", 1, dict(tc_combine_min=blocks)),
                             ("above", 1, dict(tc_combine_min=blocks + 1)), ("u64", 0, {})):
        ctx = mpc.Context(hashlib.sha256(b"combine").digest(), gemm_path=path,
                          tuning=dict(trunc_block=128, **tune))
        assert ctx.tuning()["tc_combine_min"] == tune.get("tc_combine_min", 32)
        _, pq = ctx.trunc(2, ctx.share_input(1, x), n, 13)
        ctx.profile(True)
        rc, tr = ctx.verify_trunc(3, pq, n, 13, 2, trace=True)
        assert rc == mpc.MPC_OK
        products[name] = ctx.profile_read()["k_gr_matmul"][1]
        out[name] = mpc.to_u64(tr)
    for name in out:
        assert np.array_equal(out[name], out["u64"]), name
    assert products["default"] == products["at"] == products["above"] + 1
