"""What a pipeline stage has this codec do, as cases for timing.

A case is one call pattern of the two codec classes that a stage keeps per boundary (``boundary.TahqCodec`` for
activations, ``boundary.QNaiveCodec`` for gradients), over the range of shapes, element types and options the
library takes.  ``trip`` is encode followed by decode of what was encoded (the two ends of one boundary, here on
one GPU); ``encode`` and ``decode`` are the two ends by themselves.
"""
from __future__ import annotations

import torch

from paper_2506_01352_b200.boundary import QNaiveCodec, TahqCodec

DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}


def tahq(name, way, samples, seq, hidden, dtype, tile=64, budget=3800, alloc=0, stochastic=False, outliers=0.005):
    """Activations through the TAH-Quant codec; a ranking group is one sample; outliers = share of x50 channels."""
    return dict(name=name, codec="tahq", way=way, samples=samples, seq=seq, hidden=hidden, dtype=dtype, tile=tile,
                budget=budget, alloc=alloc, stochastic=stochastic, outliers=outliers)


def qnaive(name, way, samples, seq, hidden, dtype, bits, per_tensor=False, prescale=1.0):
    """Activation gradients through the fixed-point codec of the backward half."""
    return dict(name=name, codec="qnaive", way=way, samples=samples, seq=seq, hidden=hidden, dtype=dtype, bits=bits,
                per_tensor=per_tensor, prescale=prescale)


def listed():
    return [
        # a tiny micro-batch: nothing but the latency of the call
        tahq("tiny_trip", "trip", 2, 64, 256, "f32", tile=32, budget=4000, outliers=0.016),
        # GPT-2-small-shaped boundary in fp32 at the paper's 80 % INT4 + 20 % INT3: sender, then receiver
        tahq("gpt2s_encode", "encode", 8, 1024, 768, "f32", outliers=0.01),
        tahq("gpt2s_decode", "decode", 8, 1024, 768, "f32", outliers=0.01),
        # sequences of odd length at the GPT2-XL width (25 tiles to a token): no ranking group is a whole number of units
        tahq("ragged_trip", "trip", 5, 1013, 1600, "bf16"),
        # stochastic rounding, at the same width with full sequences
        tahq("stochastic_encode", "encode", 4, 1024, 1600, "bf16", stochastic=True),
        # the LLaMA-7B-shaped boundary: the framework's headline workload
        tahq("llama7b_trip", "trip", 4, 2048, 4096, "bf16"),
        # wide tiles, one long sample, the threshold in the dense part of the scores
        tahq("wide_tile_encode", "encode", 1, 4096, 4096, "bf16", tile=128, budget=3500),
        # token-level bit allocation (A = C)
        tahq("token_alloc_trip", "trip", 4, 1024, 2048, "bf16", alloc=2048),
        # the LLaMA-13B-shaped boundary in fp32
        tahq("llama13b_trip", "trip", 8, 2048, 5120, "f32", budget=3500, outliers=0.0016),
        # the large tensor: a gibibyte of activations, 1 % outlier channels
        tahq("large_trip", "trip", 16, 4096, 8192, "bf16", outliers=0.01),
        # the backward half: 6-bit gradients of the LLaMA-7B-shaped boundary, pre-scaled
        qnaive("llama7b_grad_trip", "trip", 4, 2048, 4096, "bf16", bits=6, prescale=1024.0),
        # 10-bit gradients of the GPT-2-small-shaped boundary in fp32
        qnaive("gpt2s_grad_trip", "trip", 8, 1024, 768, "f32", bits=10),
    ]


LARGEST = 1 << 27   # elements of a drawn case


def _spread(rng, low, high):
    """An integer of [low, high], evenly over its logarithm."""
    return min(high, int(round(low * (high / low) ** rng.random())))


def draw(rng):
    way = rng.choice(["trip", "trip", "encode", "decode"])
    dtype = rng.choice(["bf16", "bf16", "f32"])
    tile = rng.choice([64, 64, 64, 32, 128])
    hidden = tile * _spread(rng, max(1, 256 // tile), 8192 // tile)
    seq = rng.choice([128, 256, 512, 1024, 2048, 4096, _spread(rng, 16, 4096), _spread(rng, 16, 4096)])
    samples = max(1, min(_spread(rng, 1, 16), LARGEST // (seq * hidden)))
    if rng.random() < 0.25:
        case = qnaive("", way, samples, seq, hidden, dtype, bits=rng.choice([6, 6, 8, 8, 10, 4, 12]),
                      per_tensor=rng.random() < 0.2, prescale=rng.choice([1.0, 1024.0, 1000.0]))
    else:
        budget = rng.choice([3800, 3800, 3500, 3000, 4000, 2000 + 100 * rng.randrange(61)])
        alloc = hidden if rng.random() < 0.1 else 0
        case = tahq("", way, samples, seq, hidden, dtype, tile=tile, budget=budget, alloc=alloc,
                    stochastic=rng.random() < 0.1, outliers=rng.choice([0.0, 0.005, 0.01, 0.05]))
    del case["name"]
    return case


def _tensor(case, seed):
    """Activations: normal values, a log-normal scale per token, a few outlier channels.  Gradients: small normal values."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    tokens, hidden = case["samples"] * case["seq"], case["hidden"]
    x = torch.randn(tokens, hidden, generator=gen, device="cuda")
    if case["codec"] == "qnaive":
        x *= 1e-3
    else:
        x *= torch.randn(tokens, 1, generator=gen, device="cuda").exp_()
        n = int(round(case["outliers"] * hidden))
        x[:, torch.randperm(hidden, generator=gen, device="cuda")[:n]] *= 50.0
    return x.to(DTYPES[case["dtype"]])


def _codec(case):
    tokens, hidden, dtype = case["samples"] * case["seq"], case["hidden"], DTYPES[case["dtype"]]
    if case["codec"] == "qnaive":
        return QNaiveCodec(tokens, hidden, dtype, "cuda", bits=case["bits"], prescale=case["prescale"],
                           per_tensor=int(case["per_tensor"]))
    return TahqCodec(tokens, hidden, dtype, "cuda", group_tokens=case["seq"], tile=case["tile"],
                     budget_millibits=case["budget"], alloc_tile=case["alloc"], rounding=int(case["stochastic"]), seed=1)


def prepare(case, seed):
    x, codec = _tensor(case, seed), _codec(case)
    packed = codec.encode(x).clone() if case["way"] == "decode" else None   # what arrived from the other stage
    return {"way": case["way"], "x": None if case["way"] == "decode" else x, "codec": codec, "packed": packed}


def run(state):
    codec = state["codec"]
    if state["way"] == "decode":
        return codec.decode(state["packed"])
    packed = codec.encode(state["x"])
    if state["way"] == "encode":
        return packed
    return {"packed": packed, "out": codec.decode(packed)}


def work(case):
    """Each direction reads its input once and writes its output once: the tensor, and the packed buffer (codes, and
    per tile 4 bytes of scale and zero-point, a pivot byte and a bit of the map; per token a 4-byte scale)."""
    n = case["samples"] * case["seq"] * case["hidden"]
    if case["codec"] == "qnaive":
        packed = n * case["bits"] / 8 + 4 * (1 if case["per_tensor"] else case["samples"] * case["seq"])
    else:
        packed = n * case["budget"] / 8000 + n // case["tile"] * 5.125
    ways = 2 if case["way"] == "trip" else 1
    encodes, decodes = case["way"] != "decode", case["way"] != "encode"
    per_element = (4 if case["codec"] == "qnaive" else 10) * encodes + 2 * decodes
    return {"bytes": ways * (n * (2 if case["dtype"] == "bf16" else 4) + packed), "flops": per_element * n}


def tolerance(case):
    """Every width, offset, scale and code is a function of the input alone, and the decoded values of the packed
    bytes alone: the oracle fixes each rounding."""
    return "exact"
