"""The calls a speculative-decoding server makes of this library, over the sizes it makes them at.

A drafter calls the low-rank head once per draft step (one row per sequence, or one per node of
a draft tree) and takes the k best tokens with their log-probabilities; a sampler that needs the
whole distribution takes the raw logits; the standard full-rank head is the same call on an
uncompressed weight matrix.  Sizes are those of the workloads in `synth.py`, the benchmark and
the tests: hidden sizes 1024 to 8192, ranks d/16 to d/4, vocabularies of 16K to 152K tokens.

A case: op       which entry point (topk, host, static, logits, full)
        M, d, r, V, k    rows, hidden size, rank (0: full rank), vocabulary, candidates per row
        scale    factor on the logits (4: the sharpened softmax)
"""
from __future__ import annotations

import math

import torch

from paper_2605_10453_b200 import binding

DEV = "cuda:0"


def _case(op, M, d, r, V, k=10, scale=1.0, name=None):
    c = {"op": op, "M": M, "d": d, "r": r, "V": V, "k": k, "scale": scale}
    if name is not None:
        c["name"] = name
    return c


def listed():
    return [
        # one sequence, a small drafter: the call is its own latency
        _case("topk", 1, 1024, 128, 32768, name="topk_m1_small"),
        # one sequence, 8B-class head: the decode step the paper reports
        _case("topk", 1, 4096, 512, 128256, name="topk_m1"),
        # the same step where activations and candidates live on the host
        _case("host", 1, 4096, 512, 128256, name="host_m1"),
        # eight draft-tree nodes, or eight sequences
        _case("topk", 8, 4096, 512, 128256, name="topk_m8"),
        # sixteen rows over a larger vocabulary with sharpened logits
        _case("topk", 16, 5120, 640, 152064, k=8, scale=4.0, name="topk_m16_sharp"),
        # a vocabulary and a rank that fit no tile: a small GPT-style head with an odd token count
        _case("topk", 5, 2880, 360, 50257, k=20, name="topk_m5_ragged"),
        # raw logits for a sampler (temperature, nucleus), four sequences
        _case("logits", 4, 2048, 256, 128256, k=1, name="logits_m4"),
        # a batch of sequences on a large model
        _case("topk", 64, 8192, 1024, 128256, name="topk_m64"),
        # throughput: 64 sequences x 8 draft-tree nodes
        _case("topk", 512, 4096, 512, 128256, name="topk_m512"),
        # the largest call: 1024 rows, rank d/4
        _case("topk", 1024, 8192, 2048, 128256, name="topk_m1024"),
        # the standard head: one row, and the throughput batch
        _case("full", 1, 4096, 0, 128256, name="full_m1"),
        _case("full", 512, 4096, 0, 128256, name="full_m512"),
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choices(("topk", "host", "static", "logits", "full"), (60, 10, 6, 12, 12))[0]
    d = rng.choice((1024, 1536, 2048, 2560, 2880, 3072, 4096, 5120, 6144, 8192))
    r = 0 if op == "full" else d // rng.choice((16, 8, 4))
    V = _log_uniform(rng, 16000, 152064)
    ragged = rng.random() < 0.2          # a vocabulary with a few tokens added is often odd
    if not ragged:
        V = V // 64 * 64
    k = 1 if op == "logits" else _log_uniform(rng, 1, 64)
    if op == "static":
        k = min(k, binding.STATIC_MAX_K)
        V = V // 64 * 64
        r = (r + 15) // 16 * 16
    most = {"topk": 1024, "host": 64, "static": binding.STATIC_MAX_M, "logits": 256, "full": 512}[op]
    if ragged or k > 32:
        most = min(most, 128)
    M = _log_uniform(rng, 1, most)
    c = _case(op, M, d, r, V, k, rng.choice((1.0, 1.0, 4.0)))
    top = max(_cost(x) for x in listed())
    while _cost(c) > top:
        c["M"] = c["M"] // 2
    return c


def _randn(rows, cols, std, g):
    out = torch.empty((rows, cols), dtype=torch.bfloat16, device=DEV)
    for r0 in range(0, rows, 512):
        n = min(512, rows - r0)
        out[r0:r0 + n] = torch.randn((n, cols), generator=g, device=DEV) * std
    return out


def prepare(case, seed):
    """Weights, activations, output buffers and the context a serving loop keeps."""
    M, d, r, V, k = (case[x] for x in ("M", "d", "r", "V", "k"))
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    s = {"op": case["op"], "k": k}
    h = _randn(M, d, 1.0, g)
    if r:
        s["A"] = _randn(d, r, 1.0 / math.sqrt(d), g)
        s["B"] = _randn(r, V, case["scale"] / math.sqrt(r), g)
    else:
        s["W"] = _randn(d, V, case["scale"] / math.sqrt(d), g)
    if case["op"] == "host":
        s["h"] = h.cpu().pin_memory()
        s["ids"] = torch.zeros((M, k), dtype=torch.int32).pin_memory()
        s["lp"] = torch.zeros((M, k), dtype=torch.float32).pin_memory()
    elif case["op"] == "logits":
        s["h"] = h
        s["logits"] = torch.empty((M, V), dtype=torch.float32, device=DEV)
    else:
        s["h"] = h
        s["ids"] = torch.empty((M, k), dtype=torch.int32, device=DEV)
        s["lp"] = torch.empty((M, k), dtype=torch.float32, device=DEV)
    if case["op"] != "static":
        s["ctx"] = binding.Context(max_M=M, max_d=max(d, r), max_V=V, max_k=k)
    return s


def run(s):
    op = s["op"]
    if op == "topk":
        return s["ctx"].slimspec_head_topk(s["h"], s["A"], s["B"], s["k"], out_ids=s["ids"], out_logprobs=s["lp"])
    if op == "host":
        return s["ctx"].slimspec_head_topk_host(s["h"], s["A"], s["B"], s["k"], out_ids_host=s["ids"],
                                                out_logprobs_host=s["lp"])
    if op == "static":
        return binding.slimspec_head_topk_static(s["h"], s["A"], s["B"], s["k"], s["ids"], s["lp"])
    if op == "logits":
        return s["ctx"].slimspec_head_logits(s["h"], s["A"], s["B"], out_logits=s["logits"])
    return s["ctx"].fullhead_topk(s["h"], s["W"], s["k"], out_ids=s["ids"], out_logprobs=s["lp"])


def work(case):
    M, d, r, V, k = (case[x] for x in ("M", "d", "r", "V", "k"))
    weights = d * r + r * V if r else d * V
    out = 4 * M * V if case["op"] == "logits" else 8 * M * k
    return {"bytes": 2 * weights + 2 * M * d + out, "flops": 2 * M * weights}


def _cost(case):
    w = work(case)
    return max(w["bytes"], w["flops"] / 50)


def tolerance(case):
    """Four times the error seen against the same path in 64 bits.  Inputs are bf16, sums fp32; the rank-r
    code keeps 16 bits or more up to 256 rows (error 3e-6 of the result, 1.6e-5 at most) and is a bf16
    operand beyond (2e-4 and 8e-4, with logits scaled by four 1.8e-3 and 6.6e-3; up to 7 % of the tokens
    lie closer together than that and may change places)."""
    if case["r"] and case["M"] > 256:
        f = case["scale"] ** 1.5
        return {"rel": 1e-3 * f, "max": 4e-3 * f, "differ": 0.15}
    return {"rel": 1.5e-5, "max": 6e-5, "differ": 5e-3}
