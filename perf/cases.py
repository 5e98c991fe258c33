"""Timed cases of the library: what a user has it do, through `binding`'s entry points.

A case is a dict of plain values.  `op` is the entry point: "forward" (Q, K, V already projected), "fused"
(un-projected inputs, linear maps inside) or "backward" (gradients of Q, K, V, E, F).  The sizes of the listed
cases are this repository's own workloads (configs.py) plus a small call, a ragged sequence length and a
float32 problem of ordinary size; `draw` spreads over the ranges those stand for.
"""
import math

import torch

from paper_2306_15799_b200 import binding, synth
from paper_2306_15799_b200.configs import PERFORMER, RNN

_VARIANT = {"performer": PERFORMER, "rnn": RNN}
_DTYPE = {"bf16": torch.bfloat16, "fp32": torch.float32}


def _case(op, variant, B, H, N, d, k, m, io="bf16", layout="bhnd", per_head=False):
    return {"op": op, "variant": variant, "io": io, "layout": layout, "per_head": per_head,
            "B": B, "H": H, "N": N, "d": d, "k": k, "m": m if variant == "performer" else 0}


def listed():
    cases = {
        # one short sequence: a single inference request, where launches and the host path are the time
        "fwd_small": _case("forward", "performer", 1, 2, 1024, 64, 128, 128),
        # the smallest configuration: float32, as a check of a model in full precision runs it
        "fwd_fp32_tiny": _case("forward", "performer", 1, 2, 256, 32, 32, 64, io="fp32"),
        # float32 at an ordinary size: evaluation of a model kept in float32
        "fwd_fp32": _case("forward", "performer", 2, 8, 4096, 64, 256, 256, io="fp32"),
        # a length that is no multiple of anything, in the layout a model's projections leave: real documents
        "fwd_ragged": _case("forward", "performer", 2, 8, 6001, 64, 256, 256, layout="bnhd"),
        # Linformer-RNN on a batch of ordinary sequences, inference and training
        "fwd_rnn": _case("forward", "rnn", 8, 12, 4096, 64, 256, 0),
        "bwd_rnn": _case("backward", "rnn", 8, 12, 4096, 64, 256, 0),
        # Linformer-Performer with a small projection: batch inference, model layout
        "fwd_mid": _case("forward", "performer", 8, 12, 8192, 64, 128, 128, layout="bnhd"),
        # the main workload: long sequences, 256 features; inference, training, and with the linear maps inside
        "fwd_long": _case("forward", "performer", 4, 16, 16384, 64, 256, 256),
        "bwd_long": _case("backward", "performer", 4, 16, 16384, 64, 256, 256),
        "fused_long": _case("fused", "performer", 4, 16, 16384, 64, 256, 256),
        # the largest: one very long sequence with wide heads
        "fwd_largest": _case("forward", "performer", 1, 8, 131072, 128, 512, 256),
        "bwd_largest": _case("backward", "performer", 1, 8, 131072, 128, 512, 256),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(("forward", "backward", "fused"), (5, 4, 1))[0]
    io = "fp32" if rng.random() < 0.12 else "bf16"
    variant = "rnn" if rng.random() < 0.3 else "performer"
    d = rng.choice((32, 64, 128) if io == "fp32" else (64, 64, 128))
    H = rng.choice((1, 2, 4, 8, 12, 16))
    B = rng.choice((1, 1, 2, 4, 8))
    k = rng.choice((64, 128, 256, 512))
    m = rng.choice((64, 128, 192, 256, 256))
    # Sequence lengths: multiples of a tile, multiples of 8, and whatever a document comes to.  The number of
    # elements of Q is kept to half of the largest listed case's (float32: an eighth of that).
    most = (1 << 23) if io == "fp32" else (1 << 26)
    N = _log_uniform(rng, 256, max(512, min(131072, most // (B * H * d))))
    step = rng.choice((128, 8, 1))
    N = max(step, N // step * step)
    if step == 1:
        N |= 1
    per_head = op != "fused" and rng.random() < 0.1
    layout = rng.choice(("bhnd", "bnhd")) if op != "fused" else "bhnd"
    return _case(op, variant, B, H, N, d, k, m, io=io, layout=layout, per_head=per_head)


def prepare(case, seed):
    """Inputs with the distributions of synth.py, drawn on the GPU: Q, K, V ~ N(0,1) d^-1/4, E, F ~ N(0,1/k),
    W block-orthogonal; un-projected inputs ~ N(0,1) with maps that give Q, K, V the same distribution."""
    gen = torch.Generator(device="cuda").manual_seed(int(seed))
    host_gen = torch.Generator().manual_seed(int(seed))
    B, H, N, d, k, m = (case[n] for n in ("B", "H", "N", "d", "k", "m"))
    dtype = _DTYPE[case["io"]]

    def normal(shape, scale):
        return torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32).mul_(scale).to(dtype)

    state = {"case": case, "variant": _VARIANT[case["variant"]], "H": H}
    if case["op"] == "fused":
        dm = H * d
        state["X"] = normal((B, N, dm), 1.0)               # self-attention: one input serves all three
        for name in ("Wq", "Wk", "Wv"):
            state[name] = normal((dm, H * d), dm ** -0.5 * d ** -0.25)
    else:
        shape = (B, N, H, d) if case["layout"] == "bnhd" else (B, H, N, d)
        for name in ("Q", "K", "V"):
            state[name] = normal(shape, d ** -0.25)
        if case["op"] == "backward":
            state["dO"] = normal(shape, 1.0)
    for name in ("E", "F"):
        state[name] = normal((H, k, N) if case["per_head"] else (k, N), k ** -0.5)
    state["W"] = synth.block_orthogonal_features(m, d, host_gen).to(dtype).cuda() if m else None
    return state


def run(state):
    s, op = state, state["case"]["op"]
    if op == "forward":
        return binding.flurka_forward(s["Q"], s["K"], s["V"], s["E"], s["F"], s["W"], s["variant"],
                                      layout=s["case"]["layout"])
    if op == "fused":
        return binding.flurka_forward_fused(s["X"], s["X"], s["X"], s["E"], s["F"], s["Wq"], s["Wk"], s["Wv"], s["W"],
                                            s["variant"], s["H"])
    return binding.flurka_backward(s["Q"], s["K"], s["V"], s["E"], s["F"], s["W"], s["dO"], s["variant"],
                                   layout=s["case"]["layout"])


def work(case):
    """Multiply-adds counted as two operations; every input read once, every output written once."""
    B, H, N, d, k, m = (case[n] for n in ("B", "H", "N", "d", "k", "m"))
    s = 4 if case["io"] == "fp32" else 2
    performer = case["variant"] == "performer"
    BH = B * H
    ef = 2 * k * N * (H if case["per_head"] else 1)
    p = m if performer else d
    if case["op"] == "backward":
        flops = BH * (12 * N * k * d + (8 * N * p * d + 12 * k * p * d if performer else 4 * N * p * d + 6 * k * p * d))
        return {"bytes": (7 * BH * N * d + 2 * ef + m * d) * s, "flops": flops}
    # feature map and product, on the N queries and on the k projected keys
    flops = BH * (N + k) * p * d * (4 if performer else 2)
    if case["op"] == "fused":
        dm = H * d
        flops += B * (4 * N * k * dm + 2 * N * dm * H * d + 4 * k * dm * H * d)
        return {"bytes": (B * N * dm + BH * N * d + ef + 3 * dm * H * d + m * d) * s, "flops": flops}
    return {"bytes": (4 * BH * N * d + ef + m * d) * s, "flops": flops + BH * 4 * N * k * d}


def tolerance(case):
    """bf16: the rounding of inputs to the second products and of the results.  float32: the exponents of the
    feature map reach |k'|^2 / 2 of a thousand and more, so 2^-24 of them is 1e-4 of a weight; the gradients
    add sums over all positions and one cancelling difference."""
    if case["io"] == "fp32":
        return {"rel": 1e-3 if case["op"] == "backward" else 1e-4}
    return {"rel": 1e-2}
