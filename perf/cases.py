"""Timed cases of the library's public calls (paper_2411_09287_gb300.mpc.Context and the models).

A case is one verified protocol step, or one whole model pass, on sharings that already sit on the
device.  Every pass of a state repeats the same protocol run (same seed, same call ids), so its
outputs repeat word for word: share components, opened values and the verification transcript.

Kinds:
  product  share X, Pi_Inner + Pi_Trunc^13 with a resident W, both verification batches, Pi_Rec
  conv     convolution (im2col inside the library) + Pi_Trunc^13 and both verification batches
  mult     elementwise Pi_Mult, Pi_MultVerify, Pi_Rec
  trunc    Pi_Trunc^t of a sharing and its verification batch
  relu     ReLU with its four verification batches
  pool     2x2 max-pool with its four verification batches
  mlp      a whole 784-128-128-10 inference, host images in, opened logits out
"""
from __future__ import annotations

import hashlib

import numpy as np
import torch

from paper_2411_09287_gb300 import mpc, secure_mlp

FRAC = 13                       # fixed-point bits of every workload of the repository
MLP_SIZES = (784, 128, 128, 10)


def listed():
    return [
        # the small plain-protocol product (64 x 128 by 128 x 64): latency and launches
        {"name": "product_64", "kind": "product", "M": 64, "N": 64, "K": 128, "words": "fixed", "keyed": False},
        # odd, ragged sizes: a packed serving batch, whose truncation bits are keyed by row
        {"name": "product_odd_keyed", "kind": "product", "M": 1501, "N": 700, "K": 1003, "words": "fixed", "keyed": True},
        # the skinny layer of the secure GEMM sweep: a large batch through a narrow layer
        {"name": "product_skinny", "kind": "product", "M": 16384, "N": 256, "K": 4096, "words": "uniform", "keyed": False},
        # a large square layer of the secure GEMM sweep
        {"name": "product_4096", "kind": "product", "M": 4096, "N": 4096, "K": 4096, "words": "uniform", "keyed": False},
        # the second convolution of Net A (16 channels 12 x 12, 5 x 5 to 16) at batch 64
        {"name": "conv_net_a", "kind": "conv", "B": 64, "C": 16, "H": 12, "k": 5, "pad": 0, "out": 16},
        # the small plain-protocol multiplication of two 4096-vectors
        {"name": "mult_4096", "kind": "mult", "n": 4096},
        # the large batch of the multiplication-verification runs
        {"name": "mult_2pow20", "kind": "mult", "n": 1 << 20},
        # standalone truncation of an odd number of values
        {"name": "trunc_100003", "kind": "trunc", "n": 100003, "t": FRAC},
        # ReLU of one image's hidden layer: the smallest serving request
        {"name": "relu_128", "kind": "relu", "n": 128},
        # ReLU of a hidden layer at batch 128
        {"name": "relu_16384", "kind": "relu", "n": 128 * 128},
        # Net A's first max-pool: one call of whole channel planes (about 2^16 comparisons)
        {"name": "pool_151x24x24", "kind": "pool", "planes": 151, "H": 24, "W": 24},
        # a whole inference of the fully connected network at batch 128
        {"name": "mlp_128", "kind": "mlp", "B": 128},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def draw(rng):
    kind = rng.choice(["product", "product", "conv", "mult", "trunc", "relu", "pool", "mlp"])
    if kind == "product":   # at most the operations and the outputs of the largest listed product
        while True:
            M, N, K = (_log_uniform(rng, 8, hi) for hi in (16384, 4096, 4096))
            if M * N <= 1 << 24 and M * K <= 1 << 26:
                return {"kind": kind, "M": M, "N": N, "K": K,
                        "words": rng.choice(["fixed", "uniform"]), "keyed": rng.random() < 0.5}
    if kind == "conv":
        return {"kind": kind, "B": _log_uniform(rng, 1, 128), "C": rng.choice([1, 3, 16, 33]),
                "H": rng.randint(8, 28), "k": rng.choice([3, 5]), "pad": rng.choice([0, 1]),
                "out": rng.randint(7, 64)}
    if kind == "mult":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 1 << 20)}
    if kind == "trunc":
        return {"kind": kind, "n": _log_uniform(rng, 1000, 1 << 20), "t": rng.choice([8, FRAC, 20])}
    if kind == "relu":
        return {"kind": kind, "n": _log_uniform(rng, 50, 1 << 16)}
    if kind == "pool":
        return {"kind": kind, "planes": _log_uniform(rng, 4, 151), "H": 2 * rng.randint(2, 12),
                "W": 2 * rng.randint(2, 12)}
    return {"kind": kind, "B": _log_uniform(rng, 1, 256)}


# ---- inputs -------------------------------------------------------------------------------------
def _words(gen, n, words):
    """n words: uniform 64-bit, or values in [-4, 4) at 13 fractional bits."""
    if words == "uniform":
        lo = torch.randint(0, 1 << 32, (n,), generator=gen, device="cuda", dtype=torch.int64)
        hi = torch.randint(0, 1 << 32, (n,), generator=gen, device="cuda", dtype=torch.int64)
        return (hi << 32) | lo
    return torch.randint(-4 << FRAC, 4 << FRAC, (n,), generator=gen, device="cuda",
                         dtype=torch.int64)


def _generator(seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    return gen


def _activations(gen, n):
    """Layer outputs before a ReLU or a pool: normal values at 13 fractional bits."""
    x = torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    return torch.floor(x * (1 << FRAC)).to(torch.int64)


def _plain(case, seed):
    """The plaintext inputs of a case."""
    gen = _generator(seed)
    k = case["kind"]
    if k == "product":
        return {"x": _words(gen, case["M"] * case["K"], case["words"]),
                "w": _words(gen, case["K"] * case["N"], case["words"])}
    if k == "conv":
        return {"x": _words(gen, case["B"] * case["C"] * case["H"] ** 2, "fixed"),
                "w": _words(gen, case["C"] * case["k"] ** 2 * case["out"], "fixed")}
    if k == "mult":
        return {"x": _words(gen, case["n"], "fixed"), "y": _words(gen, case["n"], "fixed")}
    if k == "trunc":
        return {"x": _words(gen, case["n"], "fixed") << 8}
    if k == "relu":
        return {"x": _activations(gen, case["n"])}
    if k == "pool":
        return {"x": _activations(gen, case["planes"] * case["H"] * case["W"])}
    g = np.random.default_rng(int(seed))
    return {"x": g.uniform(0.0, 1.0, (case["B"], MLP_SIZES[0])),
            "w": [g.normal(0.0, 0.05, (a, b)) for a, b in zip(MLP_SIZES, MLP_SIZES[1:])]}


def prepare(case, seed):
    p = _plain(case, seed)
    ctx = mpc.Context(hashlib.sha256(f"perf-{int(seed)}".encode()).digest())
    s = {"case": case, "ctx": ctx, "keys": None}
    k = case["kind"]
    if k == "product":
        s["x"] = p["x"]
        s["w"] = ctx.share_input(1, p["w"])
        if case["keyed"]:   # requests of 1, 2, 3, ... rows packed into one batch
            seg, left, q = [], case["M"], 0
            while left:
                rows = min(left, 1 + q % 37)
                seg.append((q, rows))
                left -= rows
                q += 1
            s["keys"] = mpc.segment_row_keys(seg, 0, 1)
    elif k == "conv":
        s["x"] = ctx.share_input(2, p["x"])
        s["w"] = ctx.share_input(1, p["w"])
        s["geom"] = (case["B"], case["C"], case["H"], case["H"], case["k"], case["k"], 1, case["pad"])
    elif k == "mult":
        s["x"], s["y"] = ctx.share_input(1, p["x"]), ctx.share_input(2, p["y"])
    elif k == "mlp":
        s["x"], s["w"] = p["x"], p["w"]
        s["shared"] = secure_mlp.share_weights(ctx, p["w"], FRAC)
    else:
        s["x"] = ctx.share_input(1, p["x"])
    torch.cuda.synchronize()
    return s


# ---- one pass -----------------------------------------------------------------------------------
def _accepted(code):
    if code != mpc.MPC_OK:
        raise RuntimeError(f"verification: {code}")


def run(state):
    c, ctx = state["case"], state["ctx"]
    k = c["kind"]
    if k == "product":
        M, N, K = c["M"], c["N"], c["K"]
        xs = ctx.share_input(2, state["x"])
        zpre, zout, pq = ctx.matmul(3, xs, state["w"], M, N, K, FRAC, row_keys=state["keys"])
        code, tr = ctx.verify_matmul(4, xs, state["w"], zpre, pq, M, N, K, FRAC, 3, trace=True,
                                     row_keys=state["keys"])
        _accepted(code)
        return {"pre": zpre, "out": zout, "transcript": tr,
                "opened": ctx.reconstruct(zout, M * N, to_host=False)}
    if k == "conv":
        cols, zpre, zout, pq, (M, N, K) = ctx.conv2d(3, state["x"], state["w"], state["geom"],
                                                     c["out"], FRAC)
        code, tr = ctx.verify_matmul(4, cols, state["w"], zpre, pq, M, N, K, FRAC, 3, trace=True)
        _accepted(code)
        return {"cols": cols, "pre": zpre, "out": zout, "transcript": tr}
    if k == "mult":
        z = ctx.mult(3, state["x"], state["y"], c["n"])
        code, tr = ctx.verify_mult(4, state["x"], state["y"], z, c["n"], 3, trace=True)
        _accepted(code)
        return {"out": z, "transcript": tr, "opened": ctx.reconstruct(z, c["n"], to_host=False)}
    if k == "trunc":
        out, pq = ctx.trunc(3, state["x"], c["n"], c["t"])
        code, tr = ctx.verify_trunc(4, pq, c["n"], c["t"], 3, trace=True)
        _accepted(code)
        return {"out": out, "pairs": pq, "transcript": tr}
    if k == "relu":
        code, out, tr = ctx.relu(3, 4, state["x"], c["n"], trace=True)
        _accepted(code)
        return {"out": out, "transcript": tr}
    if k == "pool":
        code, out, tr = ctx.maxpool2(3, 4, state["x"], (c["planes"], 1, c["H"], c["W"]), trace=True)
        _accepted(code)
        return {"out": out, "transcript": tr}
    return secure_mlp.secure_forward(ctx, state["x"], state["w"], FRAC,
                                     shared_weights=state["shared"], segments=[(7, c["B"])])


# ---- what a pass cannot do without ----------------------------------------------------------------
# Counted in words of 8 bytes and u64 multiply-adds (2 operations each).  A sharing is 6 words an
# element.  Products: P0 multiplies once, P1 and P2 twice.  Verification: every share word that
# enters a batch is weighted by its element of GR(2^64, 64) (64 multiply-adds) once.
def _product_work(M, N, K):
    E = M * N
    words = 6 * (M * K + K * N) + 2 * 6 * E + 12 * E
    macs = 5 * E * K + 64 * (6 * (M * K + K * N + E) + 12 * E)
    return words, macs


def _select_work(n):
    """A comparison and selection: 64 + 3 multiplications, one inner product of 64, 125 AND gates."""
    return 12 * n, n * (2 * (64 + 3 + 64) * 5 + 64 * 18 * (64 + 3 + 64))


def work(case):
    k = case["kind"]
    if k == "product":
        w, m = _product_work(case["M"], case["N"], case["K"])
        w += case["M"] * case["K"] + case["M"] * case["N"]
    elif k == "conv":
        ho = case["H"] + 2 * case["pad"] - case["k"] + 1
        w, m = _product_work(case["B"] * ho * ho, case["out"], case["C"] * case["k"] ** 2)
        w += 6 * case["B"] * case["C"] * case["H"] ** 2
    elif k == "mult":
        w, m = 19 * case["n"], case["n"] * (5 + 64 * 18)
    elif k == "trunc":
        w, m = 24 * case["n"], case["n"] * 64 * 12
    elif k == "relu":
        w, m = _select_work(case["n"])
    elif k == "pool":
        w, m = _select_work(3 * case["planes"] * (case["H"] // 2) * (case["W"] // 2))
    else:
        w = m = 0
        for i, (a, b) in enumerate(zip(MLP_SIZES, MLP_SIZES[1:])):
            dw, dm = _product_work(case["B"], b, a)
            w, m = w + dw, m + dm
            if i + 2 < len(MLP_SIZES):
                dw, dm = _select_work(case["B"] * b)
                w, m = w + dw, m + dm
    return {"bytes": 8 * w, "flops": 2 * m}


def exact(case, seed):
    """The values that do not depend on the protocol's randomness: opened products, and the
    network's logits in float64 for the inputs and weights that the fixed-point encoding holds."""
    if case["kind"] == "mult":
        p = _plain(case, seed)
        return {"out": None, "transcript": None, "opened": p["x"] * p["y"]}
    if case["kind"] != "mlp":
        return None
    p = _plain(case, seed)
    h = np.floor(p["x"] * (1 << FRAC)) / (1 << FRAC)
    for i, w in enumerate(p["w"]):
        h = h @ (np.floor(w * (1 << FRAC)) / (1 << FRAC))
        if i + 1 < len(p["w"]):
            h = np.maximum(h, 0.0)
    return h
