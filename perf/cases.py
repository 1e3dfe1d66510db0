"""The calls that are timed, and what each of them computes and moves at the least.

A case is one call through `paper_2609_10937_b200.binding`, the way a program calls it: bf16 CUDA tensors in hand, the
output allocated by the call.  Four kinds:

  attn     forward(q, k, v, causal=...)      prefill: every query row of B sequences of H heads
  qk       forward_qk(q, k, v)               Lq query rows against Lk keys: a decoding step, or a block of a longer prefill
  gemm     gemm(a, b, b_layout=...)          C = A B ("kn") or A B^T ("nk")
  softmax  softmax_rows(s, scale)            row softmax of a score matrix

`listed()` names twelve of them and `draw()` gives others of the same ranges.
"""
import math

import torch

from paper_2609_10937_b200 import binding


def listed():
    return [
        # The smallest call: one head, two query sub-tiles, two key steps.  Launch and host latency are what it costs.
        {"name": "attn_smallest", "kind": "attn", "B": 1, "H": 1, "Lq": 256, "Lk": 256, "d": 64, "causal": False, "var": 1},
        # An ordinary single sequence of four heads with large logits (variance 3): fewer Q tiles than SMs.
        {"name": "attn_four_heads", "kind": "attn", "B": 1, "H": 4, "Lq": 4096, "Lk": 4096, "d": 128, "causal": False, "var": 3},
        # The paper's headline shape: one long head, whose keys are shared out over the machine.
        {"name": "attn_long_head", "kind": "attn", "B": 1, "H": 1, "Lq": 16384, "Lk": 16384, "d": 128, "causal": False, "var": 1},
        # Prefill batches of a language model, wide heads and narrow ones (the narrow one is the largest case).
        {"name": "prefill_d128", "kind": "attn", "B": 4, "H": 32, "Lq": 4096, "Lk": 4096, "d": 128, "causal": False, "var": 1},
        {"name": "prefill_d64", "kind": "attn", "B": 4, "H": 32, "Lq": 8192, "Lk": 8192, "d": 64, "causal": False, "var": 1},
        # Causal prefill: the batch, and two sequences of a length that no tile divides.
        {"name": "prefill_causal_d128", "kind": "attn", "B": 4, "H": 32, "Lq": 4096, "Lk": 4096, "d": 128, "causal": True, "var": 1},
        {"name": "causal_ragged_d64", "kind": "attn", "B": 2, "H": 16, "Lq": 1111, "Lk": 1111, "d": 64, "causal": True, "var": 1},
        # A decoding step of eight sequences: one query row per head against 4096 keys and values.
        {"name": "decode_one_row", "kind": "qk", "B": 8, "H": 32, "Lq": 1, "Lk": 4096, "d": 128, "causal": False, "var": 1},
        # Matrix products: the square one, and sizes that no tile divides.
        {"name": "gemm_square", "kind": "gemm", "batch": 1, "M": 4096, "N": 4096, "K": 4096, "layout": "kn"},
        {"name": "gemm_odd", "kind": "gemm", "batch": 1, "M": 5000, "N": 3000, "K": 1000, "layout": "nk"},
        # Row softmax of the scores of one long head, and of many short sequences.
        {"name": "softmax_wide", "kind": "softmax", "rows": 8192, "cols": 8192, "d": 128},
        {"name": "softmax_short_rows", "kind": "softmax", "rows": 32768, "cols": 520, "d": 64},
    ]


_MOST_FLOPS = 4.0 * 4 * 32 * 8192 * 8192 * 64     # the largest listed case
_MOST_VALUES = 1 << 28                            # of one tensor


def _log(rng, lo, hi):
    """An integer from lo to hi, spread evenly over the logarithm."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(("attn", "attn", "attn", "qk", "gemm", "softmax"))
    while True:
        if kind in ("attn", "qk"):
            case = {"kind": kind, "B": rng.randint(1, 8), "H": _log(rng, 1, 32), "d": rng.choice((64, 128)), "var": rng.choice((1, 1, 3))}
            if kind == "attn":
                case["Lq"] = case["Lk"] = _log(rng, 128, 16384)
                case["causal"] = rng.random() < 0.5
            else:
                case["Lq"], case["Lk"], case["causal"] = _log(rng, 1, 4096), _log(rng, 256, 16384), False
            if rng.random() < 0.5:                # half of them with the usual lengths: multiples of 128
                case["Lk"] = -(-case["Lk"] // 128) * 128
                case["Lq"] = case["Lk"] if kind == "attn" else case["Lq"]
            heads = case["B"] * case["H"]
            if 4.0 * heads * case["Lq"] * case["Lk"] * case["d"] <= _MOST_FLOPS and heads * case["Lk"] * case["d"] <= _MOST_VALUES:
                return case
        elif kind == "gemm":
            case = {"kind": kind, "batch": rng.choice((1, 1, 2, 4)), "M": _log(rng, 64, 8192), "N": 8 * _log(rng, 8, 1024),
                    "K": 8 * _log(rng, 8, 1024), "layout": rng.choice(("kn", "nk"))}
            if case["batch"] * case["M"] * case["N"] <= _MOST_VALUES and 2.0 * case["batch"] * case["M"] * case["N"] * case["K"] <= _MOST_FLOPS:
                return case
        else:
            case = {"kind": kind, "rows": _log(rng, 256, 131072), "cols": 8 * _log(rng, 16, 4096), "d": rng.choice((64, 128))}
            if case["rows"] * case["cols"] <= _MOST_VALUES:
                return case


def _normal(gen, shape, std=1.0):
    """Normal values, drawn in fp32 and rounded once to bf16."""
    return (torch.randn(shape, generator=gen, device="cuda", dtype=torch.float32) * std).to(torch.bfloat16)


def prepare(case, seed):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    if case["kind"] in ("attn", "qk"):
        lead, std = (case["B"], case["H"]), math.sqrt(case["var"])
        q = _normal(gen, lead + (case["Lq"], case["d"]), std)
        k = _normal(gen, lead + (case["Lk"], case["d"]), std)
        v = _normal(gen, lead + (case["Lk"], case["d"]))
        return {"kind": case["kind"], "q": q, "k": k, "v": v, "causal": case["causal"]}
    if case["kind"] == "gemm":
        b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
        lead = (b,) if b > 1 else ()
        return {"kind": "gemm", "a": _normal(gen, lead + (M, K)), "layout": case["layout"],
                "b": _normal(gen, lead + ((K, N) if case["layout"] == "kn" else (N, K)))}
    # scores q.k of rows with unit variance: variance d, scaled back by 1 / sqrt(d) inside the call
    return {"kind": "softmax", "s": _normal(gen, (case["rows"], case["cols"]), math.sqrt(case["d"])), "scale": 1.0 / math.sqrt(case["d"])}


def run(state):
    kind = state["kind"]
    if kind == "attn":
        return binding.forward(state["q"], state["k"], state["v"], causal=state["causal"])
    if kind == "qk":
        return binding.forward_qk(state["q"], state["k"], state["v"])
    if kind == "gemm":
        return binding.gemm(state["a"], state["b"], b_layout=state["layout"])
    return binding.softmax_rows(state["s"], state["scale"])


def work(case):
    """Every input read once, every output written once; the products of the (query, key) pairs that count (causal:
    those with the key not after the query)."""
    if case["kind"] in ("attn", "qk"):
        heads, Lq, Lk, d = case["B"] * case["H"], case["Lq"], case["Lk"], case["d"]
        pairs = Lq * (Lq + 1) / 2 if case["causal"] else Lq * Lk
        return {"bytes": 2.0 * heads * d * (2 * Lq + 2 * Lk), "flops": 4.0 * heads * pairs * d}
    if case["kind"] == "gemm":
        b, M, N, K = case["batch"], case["M"], case["N"], case["K"]
        return {"bytes": 2.0 * b * (M * K + K * N + M * N), "flops": 2.0 * b * M * N * K}
    values = float(case["rows"]) * case["cols"]
    return {"bytes": 4.0 * values, "flops": 4.0 * values}


def tolerance(case):
    """About four times the distance of the results from the same path in 64 bits on the same bf16 inputs.

    Attention rounds its weights and its output to bf16: 2-norm 2.3e-3 from the exact result, single values up to 2.7e-2
    of the root mean square (causal: the first rows average few values).  The products and the row softmax round only
    the output: 1.7e-3, and 3.9e-3 of the value.
    """
    return {"rel": 9e-3, "max": 0.1} if case["kind"] in ("attn", "qk") else {"rel": 7e-3, "max": 1.6e-2}
