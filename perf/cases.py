"""The calls that a user of this library makes, as cases to be timed: sizes, inputs, one pass, its work and its tolerance.

Every case goes through the public functions of `paper_2012_01114_b200.binding` (one per C entry point).  Sizes are those
of the workloads in `paper_2012_01114_b200/inputs.py` and of the tests, or generic ones between them.  `listed()` is the
fixed set, `draw(rng)` gives further cases of the same ranges.
"""
import math

import torch

from paper_2012_01114_b200 import binding

SCHEMES = {"full": binding.FULL, "symmetric": binding.SYMMETRIC, "masked": binding.MASKED}
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}


def _case(name, entry, dtype, scheme, batch, heads, n, d_k, d_model=0, residual=False):
    c = dict(entry=entry, dtype=dtype, scheme=scheme, batch=batch, heads=heads, n=n, d_k=d_k, d_model=d_model,
             residual=residual)
    return dict(c, name=name) if name else c


def listed():
    """entry: "layer" (projections + attention), "core" (q, k, v given), "block" (layer + output projection, `residual`
    adds the skip connection), "host" (the layer from and to pinned host memory)."""
    return [
        # one short sequence, one head, full precision: the smallest call anybody makes; nothing but latency
        _case("layer f32 n64", "layer", "f32", "masked", 1, 1, 64, 64, 64),
        # one short prompt of ragged length through a 12-head layer: a latency-bound call of the throughput path
        _case("layer n200", "layer", "bf16", "full", 1, 12, 200, 64, 768),
        # encoder layer over a batch of medium sequences
        _case("layer n512", "layer", "bf16", "full", 8, 12, 512, 64, 768),
        # decoder attention block (projections, masked attention, output projection, residual): one prefill step
        _case("block n1024", "block", "bf16", "masked", 8, 12, 1024, 64, 768, residual=True),
        # the layer called on host buffers, as a program without device tensors does
        _case("host n512", "host", "bf16", "full", 8, 12, 512, 64, 768),
        # many short sequences with q, k, v at hand: bound by memory traffic
        _case("core n256", "core", "bf16", "full", 256, 16, 256, 128),
        # query = key = value: the paper's first scheme at a medium length
        _case("core n1024 symmetric", "core", "bf16", "symmetric", 64, 16, 1024, 128),
        # long ragged sequences, head size between the tile widths
        _case("core n3001 d96", "core", "bf16", "masked", 2, 16, 3001, 96),
        # long-context prefill: the largest masked call
        _case("core n8192", "core", "bf16", "masked", 2, 16, 8192, 128),
        # few wide heads
        _case("core n2048 d256", "core", "bf16", "masked", 4, 8, 2048, 256),
        # full-precision layer over a small batch
        _case("layer f32 n512", "layer", "f32", "full", 4, 12, 512, 64, 768),
        # full-precision core, masked, the longest sequence that path takes
        _case("core f32 n1024", "core", "f32", "masked", 2, 8, 1024, 128),
    ]


# What limits a drawn case: its work stays within half of that of the largest listed case of its kind (masked n = 8192 in
# bf16, symmetric n = 1024, the fp32 layer at n = 512), so that it takes no longer at a size that runs less well, and its
# tensors within 256 MB each (bf16).
_MOST_FLOPS = {"bf16": 2.7e11, "symmetric": 2.0e11, "f32": 5.0e9}
_MOST_ELEMENTS = 1 << 27


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: entry, type, scheme and sizes over the ranges the listed cases stand for."""
    while True:
        dtype = rng.choice(["bf16", "bf16", "bf16", "f32"])
        entry = rng.choice(["layer", "layer", "block", "core", "core", "core", "host"])
        scheme = rng.choice(["full", "full", "masked", "masked", "symmetric"])
        heads = rng.choice([1, 2, 4, 8, 12, 16, 20, 32])
        if dtype == "f32":
            n, d_k = _log_int(rng, 16, 1024), rng.choice([16, 20, 32, 48, 64, 64, 80, 128])
        else:
            wide = scheme != "symmetric" and rng.random() < 0.15
            n = _log_int(rng, 16, 8192)
            d_k = rng.choice([160, 192, 256]) if wide else rng.choice([32, 48, 64, 64, 80, 96, 128, 128])
        if rng.random() < 0.4:                       # lengths that are a multiple of the tile are as common as odd ones
            n = max(128, n // 128 * 128) if dtype == "bf16" or n >= 128 else n
        tokens = _log_int(rng, 64, 65536)
        batch = max(1, tokens // n)
        d_model = 0
        if entry != "core":
            if dtype == "bf16" and heads * d_k % 64:
                continue
            d_model = max(64, heads * d_k // 64 * 64)
            if rng.random() < 0.3:
                d_model = rng.choice([64, 192, 320, 768, 1024])
        c = _case(None, entry, dtype, scheme, batch, heads, n, d_k, d_model, entry == "block" and rng.random() < 0.5)
        kind = "f32" if dtype == "f32" else ("symmetric" if scheme == "symmetric" else "bf16")
        if work(c)["flops"] > _MOST_FLOPS[kind] or batch * n * max(heads * d_k, d_model) > _MOST_ELEMENTS:
            continue
        if entry == "host" and batch * n * max(heads * d_k, d_model) > 1 << 23:     # pinned buffers of 16 MB (bf16)
            continue
        return c


def prepare(case, seed):
    """Inputs N(0, 1) (activations, q, k, v) and N(0, 1) / sqrt(fan-in) (weights), and the output buffer such a program
    keeps; for "host" all of them in pinned host memory."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    dt = DTYPES[case["dtype"]]
    B, H, n, d, D = case["batch"], case["heads"], case["n"], case["d_k"], case["d_model"]
    sym = case["scheme"] == "symmetric"

    def normal(shape, scale=1.0):
        t = torch.empty(shape, dtype=dt, device="cuda").normal_(0.0, scale, generator=g)
        return torch.empty(shape, dtype=dt, pin_memory=True).copy_(t) if case["entry"] == "host" else t

    s = {"case": case, "scheme": SCHEMES[case["scheme"]], "heads": H}
    if case["entry"] == "core":
        s["in"] = [normal((B, n, H, d)) for _ in range(1 if sym else 3)] + ([None, None] if sym else [])
        s["out"] = torch.empty((B, n, H * d), dtype=dt, device="cuda")
        return s
    s["in"] = [normal((B, n, D))] + [normal((D, H * d), D ** -0.5) for _ in range(1 if sym else 3)] + ([None, None] if sym else [])
    if case["entry"] == "block":
        s["Wo"] = normal((H * d, D), (H * d) ** -0.5)
    width = D if case["entry"] == "block" else H * d
    s["out"] = torch.empty((B, n, width), dtype=dt, pin_memory=True) if case["entry"] == "host" else \
        torch.empty((B, n, width), dtype=dt, device="cuda")
    return s


def run(s):
    """One call of the public entry point; returns the whole output."""
    entry = s["case"]["entry"]
    if entry == "core":
        return binding.psa_attention_core(*s["in"], s["scheme"], out=s["out"])
    if entry == "block":
        return binding.psa_attention_block(*s["in"], s["Wo"], s["heads"], s["scheme"], out=s["out"],
                                           residual=s["in"][0] if s["case"]["residual"] else None)
    if entry == "host":
        return binding.psa_attention_host(*s["in"], s["heads"], s["scheme"], s["out"])
    if s["case"]["dtype"] == "f32":
        return binding.psa_attention_f32(*s["in"], s["heads"], s["scheme"], out=s["out"])
    return binding.psa_attention(*s["in"], s["heads"], s["scheme"], out=s["out"])


def work(case):
    """Element-level operations of the scheme (two per multiply-accumulate) and every input and output once."""
    B, H, n, d, D = case["batch"], case["heads"], case["n"], case["d_k"], case["d_model"]
    es = 2 if case["dtype"] == "bf16" else 4
    tri = n * (n + 1) // 2
    macs = B * H * d * ((n * n if case["scheme"] == "full" else tri) + (tri if case["scheme"] == "masked" else n * n))
    tensors = 1 if case["scheme"] == "symmetric" else 3
    if case["entry"] == "core":
        elements = (tensors + 1) * B * n * H * d
    else:
        macs += tensors * B * n * D * H * d
        elements = B * n * D + tensors * D * H * d + B * n * H * d
        if case["entry"] == "block":
            macs += B * n * D * H * d
            elements += D * H * d + B * n * (D - H * d)         # Wo; the output has D columns; a residual is X itself
    return {"bytes": float(es * elements), "flops": 2.0 * macs}


def tolerance(case):
    """Four times what the path is off from its own result in 64 bits, measured over listed and drawn cases: bf16 (inputs,
    weights of the softmax and outputs rounded to 8 bits) rel 1.7e-3 .. 3.6e-3, max 4e-3 .. 6e-2; fp32 rel 3e-7 .. 1e-6,
    max 3e-6 .. 8e-6."""
    return {"rel": 1e-2, "max": 0.25} if case["dtype"] == "bf16" else {"rel": 4e-6, "max": 4e-5}
