"""The workloads on which the speed of the attention forward is measured.

Everything goes through ``binding.attn_fwd``, the entry point a user's program calls.  The listed
cases cover what such a program does with it: prefill of short, middle and long sequences, a chunk
of new queries against a long context, and decoding one new token; 16-bit and fp8 storage; head
dimensions 64 and 128; grouped heads; causal and full attention; the three weight maps in earnest
use.  Shapes are those of the workload descriptions, tests and benchmark of this repository, or
generic ones of the same ranges.

Inputs are N(0,1) draws in the order q, k, v (with ``peaked`` every key row is multiplied by its own
U(0.5, 2) factor), cast to the storage type; fp8 tensors are quantised with a per-tensor descale
amax / 448.  They are made on the GPU from a seeded generator.
"""
import math

import numpy as np
import torch

from paper_2609_33586_b200 import binding

DTYPES = {"bf16": torch.bfloat16, "fp16": torch.float16, "fp8_e4m3": torch.float8_e4m3fn}
E4M3_MAX = 448.0


def _case(name, B, Hq, Hkv, Sq, Sk, D, causal, dtype, mode, peaked=False):
    return {"name": name, "B": B, "Hq": Hq, "Hkv": Hkv, "Sq": Sq, "Sk": Sk, "D": D, "causal": causal,
            "dtype": dtype, "mode": mode, "peaked": peaked}


def listed():
    return [
        # the smallest configuration: latency of one call
        _case("tiny_causal_bf16_d64", 1, 2, 2, 256, 256, 64, True, "bf16", "h15"),
        # a short prompt: one sequence of 1K tokens, fp8
        _case("causal_1k_fp8", 1, 16, 16, 1024, 1024, 128, True, "fp8_e4m3", "h15"),
        # the model-fidelity shape: a small batch of 2K prompts, grouped heads 12 / 2, peaked rows
        _case("gqa_causal_2k_bf16", 4, 12, 2, 2048, 2048, 128, True, "bf16", "h15", True),
        # cross attention of two ragged lengths, full attention, the exact softmax
        _case("cross_ragged_bf16", 3, 12, 2, 1337, 2803, 128, False, "bf16", "exact"),
        # head dimension 64, IEEE half, an odd length, power-of-two weights
        _case("causal_3001_fp16_d64_pot", 2, 16, 16, 3001, 3001, 64, True, "fp16", "pot"),
        # a long prompt in 16-bit storage with the exact softmax
        _case("causal_8k_bf16_exact", 1, 16, 16, 8192, 8192, 128, True, "bf16", "exact"),
        # the headline: causal 8K prefill on fp8
        _case("causal_8k_fp8", 2, 16, 16, 8192, 8192, 128, True, "fp8_e4m3", "h15"),
        # its full-attention twin with the exact softmax
        _case("noncausal_8k_fp8_exact", 2, 16, 16, 8192, 8192, 128, False, "fp8_e4m3", "exact"),
        # the largest: one 16K prompt, grouped heads 32 / 8
        _case("causal_16k_gqa_bf16", 1, 32, 8, 16384, 16384, 128, True, "bf16", "h15"),
        # chunked prefill: 512 new queries against a 16K context
        _case("chunk_512_of_16k_bf16", 1, 32, 8, 512, 16384, 128, True, "bf16", "h15"),
        # decoding: one new token for each of four sequences with 16K of context
        _case("decode_b4_16k_bf16", 4, 32, 8, 1, 16384, 128, True, "bf16", "h15"),
        # decoding one sequence with 8K of context, fp8 cache, the exact softmax
        _case("decode_b1_8k_fp8_exact", 1, 32, 8, 1, 8192, 128, True, "fp8_e4m3", "exact"),
    ]


# No drawn case costs more multiply-adds, or more bytes, than the largest listed ones.
_MOST_FLOPS = 4.0 * 32 * 128 * (16384 * 16385 / 2)
_MOST_BYTES = 300e6


def _length(rng, low, high):
    """A length between low and high, spread over its logarithm: any number, or rounded to a multiple of 128."""
    n = int(round(math.exp(rng.uniform(math.log(low), math.log(high)))))
    if rng.random() < 0.4:
        n = (n + 64) // 128 * 128
    return min(max(n, low), high)


def draw(rng):
    while True:
        Hq, Hkv = rng.choice([(2, 2), (12, 2), (16, 16), (16, 4), (32, 8), (32, 32)])
        D = rng.choice([128, 128, 64])
        dtype = rng.choice(["bf16", "bf16", "fp8_e4m3", "fp8_e4m3", "fp16"])
        mode = rng.choice(["h15", "h15", "exact", "exact", "pot"])
        peaked = rng.random() < 0.2
        kind = rng.choice(["prefill", "prefill", "prefill", "cross", "chunk", "decode"])
        B = rng.choice([1, 1, 2, 3, 4])
        causal = True
        if kind == "prefill":       # a prompt against itself
            Sq = Sk = _length(rng, 128, 16384)
            causal = rng.random() < 0.75
        elif kind == "cross":       # two lengths of their own, full attention
            Sq, Sk = _length(rng, 64, 8192), _length(rng, 64, 8192)
            causal = False
        elif kind == "chunk":       # new queries at the end of a longer context
            Sk = _length(rng, 1024, 32768)
            Sq = _length(rng, 16, 1024)
        else:                       # decode: one new token, or a few proposed ones
            Sk = _length(rng, 128, 32768)
            Sq = rng.choice([1, 1, 1, 2, 4])
            B = rng.choice([1, 2, 4, 8, 16])
        c = {"B": B, "Hq": Hq, "Hkv": Hkv, "Sq": Sq, "Sk": Sk, "D": D, "causal": causal, "dtype": dtype, "mode": mode,
             "peaked": peaked}
        w = work(c)
        if w["flops"] <= _MOST_FLOPS and w["bytes"] <= _MOST_BYTES:
            return c


def _store(x, dtype):
    if dtype != "fp8_e4m3":
        return x.to(DTYPES[dtype]), 1.0
    descale = float(np.float32(float(x.abs().max()) / E4M3_MAX))
    return (x / descale).clamp_(-E4M3_MAX, E4M3_MAX).to(torch.float8_e4m3fn), descale


def prepare(case, seed):
    c = case
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)

    def normal(S, H):
        return torch.randn(c["B"], S, H, c["D"], generator=g, dtype=torch.float32, device="cuda")

    q, dq = _store(normal(c["Sq"], c["Hq"]), c["dtype"])
    k = normal(c["Sk"], c["Hkv"])
    v, dv = _store(normal(c["Sk"], c["Hkv"]), c["dtype"])
    if c["peaked"]:
        k *= torch.rand(c["B"], c["Sk"], c["Hkv"], 1, generator=g, device="cuda") * 1.5 + 0.5
    k, dk = _store(k, c["dtype"])
    return {"q": q, "k": k, "v": v,
            "options": {"causal": c["causal"], "softmax_scale": float(np.float32(1.0 / math.sqrt(c["D"]))),
                        "weight_mode": binding.MODES[c["mode"]], "q_descale": dq, "k_descale": dk, "v_descale": dv}}


def run(state):
    return binding.attn_fwd(state["q"], state["k"], state["v"], **state["options"])   # (O, LSE)


def work(case):
    """q, k, v read once, O (bf16) and LSE (fp32) written once; two multiply-adds of length D per visible pair."""
    c = case
    B, Sq, Sk, D = c["B"], c["Sq"], c["Sk"], c["D"]
    if c["causal"]:   # row i sees the keys up to i + Sk - Sq
        first = Sk - Sq + 1
        pairs = sum(max(0, first + i) for i in range(Sq)) if first < 1 else Sq * first + Sq * (Sq - 1) // 2
    else:
        pairs = Sq * Sk
    es = 1 if c["dtype"] == "fp8_e4m3" else 2
    return {"bytes": float(B * D * es * (Sq * c["Hq"] + 2 * Sk * c["Hkv"]) + B * Sq * c["Hq"] * (2 * D + 4)),
            "flops": 4.0 * B * c["Hq"] * D * pairs}


def tolerance(case):
    """Four times what the forward differs by from its own loop in 64 bits, on the listed cases.

    O is stored in bf16 (relative error 1.7e-3; the exact softmax with 16-bit P 2.3e-3), LSE adds nothing to that.
    ``max`` is larger in the rounding maps, where a score within an fp32 rounding of a tie may take either
    neighbour (0.18 in rows of a few keys).  The exact softmax on fp8 inputs stores P in e4m3, whose three fraction
    bits show in O (2.6e-2, max 0.14)."""
    if case["mode"] != "exact":
        return {"rel": 7e-3, "max": 0.7}
    if case["dtype"] == "fp8_e4m3":
        return {"rel": 3e-2, "max": 0.55}
    return {"rel": 9e-3, "max": 0.14}
