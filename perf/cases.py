"""The calls that programs built on this library spend their time in, as cases that can be prepared, run and timed.

The library serves transformer inference and the matrix products around it, so the cases are its entry points at the
sizes of the two transformer blocks and of the benchmark configurations in `workloads.py`: GPT-style layers (hidden
768, 12 heads of 64, MLP 3072) and Llama-3-8B-style layers (hidden 4096, 32 query heads over 8 key/value heads of
128, SwiGLU MLP 14336).  `listed()` holds one call of each kind, from the smallest to the largest; `draw()` gives
more of the same kinds over the whole range of sizes a program meets: one token to 16384, ragged sequence lengths,
odd widths, both weight layouts, BF16 and FP32 outputs, FP8 operands, grouped experts.

Values are those of the configurations: activations N(0, 1), weights N(0, 0.02^2), norm gains 1 + N(0, 0.1^2),
biases N(0, 0.02^2); square products N(0, 1) / sqrt(K), long-K products U(-1, 1).
"""
from __future__ import annotations

import math

import torch

from paper_2604_26666_b200.binding import Handle

# (inputs, outputs, epilogue) of the linear layers of the two blocks; a gated layer's weight has 2 x outputs columns
LINEARS = {
    "gpt": [(768, 2304, "BIAS"), (768, 768, "BIAS_RESIDUAL"), (768, 3072, "BIAS_GELU_TANH"), (3072, 768, "BIAS_RESIDUAL")],
    "llama": [(4096, 6144, "NONE"), (4096, 4096, "BIAS_RESIDUAL"), (4096, 14336, "SILU_GATE"), (14336, 4096, "BIAS_RESIDUAL")],
}
# (query heads, key/value heads, head dimension, MLP width)
HEADS = {"gpt": (12, 12, 64, 3072), "llama": (32, 8, 128, 14336)}
MOST_FLOPS = 3.7e12  # no drawn case asks for more than the largest listed one


def _linear(name, M, K, N, epilogue, layout="NK", bias=None):
    if bias is None:
        bias = epilogue in ("BIAS", "BIAS_RELU", "BIAS_GELU_TANH")
    return {"name": name, "op": "linear", "M": M, "K": K, "N": N, "epilogue": epilogue, "layout": layout, "bias": bias}


def listed():
    return [
        # the smallest call: one 512^3 product with bias and ReLU, where latency and launches are the time
        _linear("linear_512", 512, 512, 512, "BIAS_RELU", layout="KN"),
        # one decode step of 16 sequences through an attention output projection: the weights are read for 16 rows
        _linear("linear_decode_16", 16, 4096, 4096, "BIAS_RESIDUAL"),
        # decode attention: one new token of 32 sequences against 2000 cached ones, grouped queries
        {"name": "attention_decode_32x2000", "op": "attention", "B": 32, "Tq": 1, "Tk": 2000, "heads": "llama", "causal": False},
        # an MLP up-projection with GELU for a batch of prompts whose lengths do not add up to anything round
        _linear("linear_gelu_3001", 3001, 768, 3072, "BIAS_GELU_TANH"),
        # causal prefill of a batch of ragged prompts
        {"name": "attention_prefill_16x1000", "op": "attention", "B": 16, "Tq": 1000, "Tk": 1000, "heads": "gpt", "causal": True},
        # many independent products (per-head or per-sample)
        {"name": "gemm_batched_128", "op": "gemm_batched", "batch": 128, "M": 512, "N": 512, "K": 1024, "layout": "KN"},
        # a product with a very long K and an FP32 result (a weight gradient, a Gram matrix)
        {"name": "gemm_splitk_131072", "op": "gemm_splitk", "M": 256, "N": 256, "K": 131072, "layout": "KN"},
        # one layer of a mixture of experts: 16384 tokens routed at random to 64 small experts
        {"name": "grouped_64_experts", "op": "grouped", "groups": 64, "tokens": 16384, "K": 2048, "N": 2048,
         "epilogue": "NONE", "bias": False, "fp8": False},
        # a QKV projection on FP8 operands
        {"name": "linear_fp8_qkv", "op": "linear_fp8", "M": 8192, "K": 4096, "N": 6144, "epilogue": "NONE", "bias": False},
        # the large square product
        {"name": "gemm_8192", "op": "gemm", "M": 8192, "N": 8192, "K": 8192, "layout": "KN", "out": "bf16"},
        # whole blocks, forward: 128 sequences of 512 tokens, and 8192 tokens of a Llama-sized block
        {"name": "block_gpt_128x512", "op": "block", "kind": "gpt", "B": 128, "T": 512},
        {"name": "block_llama_4x2048", "op": "block", "kind": "llama", "B": 4, "T": 2048},
    ]


def _log(rng, lo, hi, step=1):
    """A size spread over the logarithm of [lo, hi], a multiple of `step`."""
    v = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    return max(lo, min(hi, int(round(v / step)) * step))


def draw(rng):
    for _ in range(1000):
        case = _draw(rng)
        if work(case)["flops"] <= MOST_FLOPS:
            return case
    raise RuntimeError("no case small enough was drawn")


def _draw(rng):
    op = rng.choice(["linear", "linear", "linear", "gemm", "gemm", "gemm_batched", "gemm_splitk", "grouped", "linear_fp8",
                     "prefill", "prefill", "decode", "norm", "block", "block"])
    model = rng.choice(["gpt", "llama"])
    tokens = 16384 if model == "gpt" else 8192
    if op == "linear":
        K, N, epilogue = rng.choice(LINEARS[model])
        case = _linear("", _log(rng, 1, tokens), K, N, epilogue, rng.choice(["NK", "NK", "NK", "KN"]),
                       bias=epilogue != "NONE" and model == "gpt")
        del case["name"]
        return case
    if op == "gemm":
        layout = rng.choice(["KN", "NK"])
        # a [K, N] operand has rows of N values, which have to be whole 16-byte pieces; an [N, K] one takes any N
        return {"op": "gemm", "M": _log(rng, 256, 8192), "N": _log(rng, 256, 8192, 8 if layout == "KN" else 1),
                "K": _log(rng, 256, 8192, 8), "layout": layout, "out": rng.choice(["bf16", "bf16", "f32"])}
    if op == "gemm_batched":
        return {"op": op, "batch": _log(rng, 8, 128), "M": _log(rng, 64, 512), "N": _log(rng, 64, 2048, 8),
                "K": _log(rng, 64, 1024, 8), "layout": rng.choice(["KN", "NK"])}
    if op == "gemm_splitk":
        return {"op": op, "M": _log(rng, 64, 256), "N": _log(rng, 64, 256, 8), "K": _log(rng, 16384, 524288, 8),
                "layout": rng.choice(["KN", "NK"])}
    if op == "grouped":
        K, N, epilogue, groups = rng.choice([(2048, 2048, "NONE", 64), (2048, 2048, "NONE", 32), (768, 3072, "BIAS_GELU_TANH", 8),
                                             (4096, 14336, "SILU_GATE", 8), (14336, 4096, "NONE", 8)])
        return {"op": op, "groups": groups, "tokens": _log(rng, 256, 16384), "K": K, "N": N, "epilogue": epilogue,
                "bias": epilogue.startswith("BIAS"), "fp8": rng.random() < 0.25}
    if op == "linear_fp8":
        K, N, epilogue = rng.choice([l for l in LINEARS[model] if l[2] != "BIAS_RESIDUAL"])
        return {"op": op, "M": _log(rng, 16, tokens), "K": K, "N": N, "epilogue": epilogue, "bias": epilogue.startswith("BIAS")}
    if op == "prefill":
        T = _log(rng, 64, 4096)
        return {"op": "attention", "B": _log(rng, 1, max(1, 2 * tokens // T)), "Tq": T, "Tk": T, "heads": model,
                "causal": rng.random() < 0.7}
    if op == "decode":
        Tk = _log(rng, 128, 8192)
        return {"op": "attention", "B": _log(rng, 1, 64), "Tq": 1, "Tk": Tk, "heads": model, "causal": False}
    if op == "norm":
        return {"op": op, "kind": "layer" if model == "gpt" else "rms", "M": _log(rng, 16, 4 * tokens),
                "C": 768 if model == "gpt" else 4096}
    T = _log(rng, 64, 2048)
    return {"op": "block", "kind": model, "B": _log(rng, 1, max(1, tokens // T)), "T": T}


_handles: dict = {}


def _handle() -> Handle:
    """The handle a program creates once."""
    if "h" not in _handles:
        _handles["h"] = Handle(torch.cuda.current_device())
    return _handles["h"]


def _sizes(case):
    """(B, Tq, Tk, Hq, Hkv, D) of an attention case."""
    Hq, Hkv, D, _ = HEADS[case["heads"]]
    return case["B"], case["Tq"], case["Tk"], Hq, Hkv, D


def prepare(case, seed):
    dev = torch.device("cuda", torch.cuda.current_device())
    gen = torch.Generator(device=dev).manual_seed(seed)

    def normal(shape, scale=1.0, shift=0.0):
        t = torch.randn(shape, generator=gen, device=dev, dtype=torch.bfloat16)
        return t if scale == 1.0 and shift == 0.0 else t.mul_(scale).add_(shift)

    def uniform(shape):
        return torch.rand(shape, generator=gen, device=dev, dtype=torch.float32).mul_(2.0).sub_(1.0).to(torch.bfloat16)

    def codes(shape, scale):
        """Per-tensor quantised E4M3 values: four standard deviations reach the format's 448."""
        t = torch.randn(shape, generator=gen, device=dev, dtype=torch.bfloat16).mul_(112.0).clamp_(-448.0, 448.0)
        return t.to(torch.float8_e4m3fn), scale / 112.0

    s = {"case": case, "h": _handle()}
    op = case["op"]
    if op in ("linear", "linear_fp8", "grouped"):
        gate = case["epilogue"] == "SILU_GATE"
        M, K, N = case.get("M", case.get("tokens")), case["K"], case["N"]
        Nw = 2 * N if gate else N
        groups = (case["groups"],) if op == "grouped" else ()
        if op == "linear_fp8" or case.get("fp8"):
            s["X"], sx = codes((M, K), 1.0)
            s["W"], sw = codes(groups + (Nw, K), 0.02)
            s["scale"] = sx * sw
        else:
            s["X"] = uniform((M, K)) if case["epilogue"] == "BIAS_RELU" else normal((M, K))
            s["W"] = normal(groups + ((K, Nw) if case.get("layout") == "KN" else (Nw, K)), 0.02)
        s["bias"] = normal((N,), 0.02) if case["bias"] else None
        s["residual"] = normal((M, N)) if case["epilogue"] == "BIAS_RESIDUAL" else None
        if op == "grouped":  # every token picks an expert at random
            pick = torch.randint(0, case["groups"], (M,), generator=gen, device=dev)
            s["rows"] = torch.bincount(pick, minlength=case["groups"]).tolist()
    elif op in ("gemm", "gemm_batched", "gemm_splitk"):
        b = (case["batch"],) if op == "gemm_batched" else ()
        M, N, K = case["M"], case["N"], case["K"]
        wshape = b + ((K, N) if case["layout"] == "KN" else (N, K))
        if op == "gemm_splitk":
            s["X"], s["W"] = uniform((M, K)), uniform(wshape)
        else:
            scale = K ** -0.5 if op == "gemm" else 1.0
            s["X"], s["W"] = normal(b + (M, K), scale), normal(wshape, scale)
    elif op == "attention":
        B, Tq, Tk, Hq, Hkv, D = _sizes(case)
        s["q"], s["k"], s["v"] = normal((B, Tq, Hq, D)), normal((B, Tk, Hkv, D)), normal((B, Tk, Hkv, D))
    elif op == "norm":
        C = case["C"]
        s["X"], s["gamma"] = normal((case["M"], C)), normal((C,), 0.1, 1.0)
        s["beta"] = normal((C,), 0.02) if case["kind"] == "layer" else None
    else:  # block
        kind = case["kind"]
        Hq, Hkv, D, ffn = HEADS[kind]
        C, qc = Hq * D, (Hq + 2 * Hkv) * D
        w = {"norm1_gamma": normal((C,), 0.1, 1.0), "norm2_gamma": normal((C,), 0.1, 1.0), "wqkv": normal((qc, C), 0.02),
             "wo": normal((C, C), 0.02), "w1": normal((2 * ffn if kind == "llama" else ffn, C), 0.02),
             "w2": normal((C, ffn), 0.02)}
        if kind == "gpt":
            for name, n in (("norm1_beta", C), ("norm2_beta", C), ("bqkv", qc), ("bo", C), ("b1", ffn), ("b2", C)):
                w[name] = normal((n,), 0.02)
        s["weights"] = w
        s["X"] = normal((case["B"] * case["T"], C))
        s["desc"] = s["h"].block_desc(kind, case["B"], case["T"], Hq, Hkv, D, ffn, w)
    return s


def run(state):
    case, h = state["case"], state["h"]
    op = case["op"]
    if op == "linear":
        return h.linear(state["X"], state["W"], bias=state["bias"], residual=state["residual"], epilogue=case["epilogue"],
                        layout=case["layout"])
    if op == "linear_fp8":
        return h.linear_fp8(state["X"], state["W"], state["scale"], bias=state["bias"], epilogue=case["epilogue"])
    if op == "grouped":
        if case["fp8"]:
            return h.linear_grouped_fp8(state["X"], state["W"], state["rows"], state["scale"], bias=state["bias"],
                                        epilogue=case["epilogue"])
        return h.linear_grouped(state["X"], state["W"], state["rows"], bias=state["bias"], epilogue=case["epilogue"])
    if op == "gemm":
        return h.gemm(state["X"], state["W"], layout=case["layout"],
                      out_dtype=torch.float32 if case["out"] == "f32" else torch.bfloat16)
    if op == "gemm_batched":
        return h.gemm_batched(state["X"], state["W"], layout=case["layout"])
    if op == "gemm_splitk":
        return h.gemm_splitk(state["X"], state["W"], layout=case["layout"])
    if op == "attention":
        return h.attention(state["q"], state["k"], state["v"], causal=case["causal"])
    if op == "norm":
        return h.norm(state["X"], state["gamma"], state["beta"], kind=case["kind"])
    return h.block_forward(state["desc"], state["X"])


def work(case):
    op = case["op"]
    if op in ("linear", "linear_fp8", "grouped"):
        M, K, N = case.get("M", case.get("tokens")), case["K"], case["N"]
        Nw = 2 * N if case["epilogue"] == "SILU_GATE" else N
        e = 1 if op == "linear_fp8" or case.get("fp8") else 2
        b = e * (M * K + case.get("groups", 1) * Nw * K) + 2 * M * N
        if case["epilogue"] == "BIAS_RESIDUAL":
            b += 2 * M * N
        if case["bias"]:
            b += 2 * N
        return {"bytes": b, "flops": 2 * M * Nw * K}
    if op in ("gemm", "gemm_batched", "gemm_splitk"):
        n, M, N, K = case.get("batch", 1), case["M"], case["N"], case["K"]
        out = 4 if op == "gemm_splitk" or case.get("out") == "f32" else 2
        return {"bytes": n * (2 * (M * K + K * N) + out * M * N), "flops": 2 * n * M * N * K}
    if op == "attention":
        B, Tq, Tk, Hq, Hkv, D = _sizes(case)
        pairs = Tq * (Tq + 1) // 2 if case["causal"] else Tq * Tk
        return {"bytes": 2 * B * D * (2 * Tq * Hq + 2 * Tk * Hkv), "flops": 4 * D * pairs * B * Hq}
    if op == "norm":
        return {"bytes": 4 * case["M"] * case["C"], "flops": 8 * case["M"] * case["C"]}
    kind, B, T = case["kind"], case["B"], case["T"]
    Hq, Hkv, D, ffn = HEADS[kind]
    tok, C, qc = B * T, Hq * D, (Hq + 2 * Hkv) * D
    up = 2 * ffn if kind == "llama" else ffn
    weights = qc * C + C * C + up * C + C * ffn
    # each stage reads and writes its activations once: norm, QKV, attention, projection, norm, up, down
    acts = tok * ((C + C) + (C + qc) + (qc + C) + (C + C + C) + (C + C) + (C + ffn) + (ffn + C + C))
    return {"bytes": 2 * (weights + acts), "flops": 2 * tok * weights + 4 * D * (T * (T + 1) // 2) * B * Hq}


def tolerance(case):
    """About four times the distance of the present results from the same computation in 64 bits (in brackets).
    One rounding to BF16 is what separates a product from the exact one; FP32 results carry the order of the sums over
    K; attention adds the rounding of the probabilities (`max`: first causal rows, where one of them weighs most); a
    block adds up the roundings of its seven stages."""
    op = case["op"]
    if op == "gemm_splitk" or case.get("out") == "f32":
        return {"rel": 1.5e-5, "max": 4e-5}  # (3.4e-6, 9.4e-6 at K = 131072; less for shorter sums)
    if op == "attention":
        return {"rel": 1e-2, "max": 1e-1}  # (2.5e-3, 2.6e-2)
    if op == "block":
        return {"rel": 1e-2 if case["kind"] == "gpt" else 1.8e-2, "max": 1.2e-1}  # (2.5e-3 and 4.3e-3, 2.9e-2)
    return {"rel": 7e-3, "max": 1.6e-2}  # (1.7e-3, 3.9e-3)
