"""Performance cases of the rotate-and-quantize library, as a program that serves or calibrates a model calls it.

A case names a kind of call and its sizes:

  quantize    activations or KV entries -> packed codes and scales (Plan.rotate_quantize)
  dequantize  packed codes and scales -> bf16 or fp32 rows, rotated back or left in the rotated domain (Plan.dequantize)
  linear      one layer: activations -> codes -> output from the packed codes of both sides (Plan.rotate_quantize, then
              Plan.quantized_matmul); the weights are quantized once, beforehand
  clip        K candidate clip ratios scored by quantization error (Plan.clip_error)

Rows are tokens, or KV entries (one per token and head).  Widths are the ones of the configurations in
paper_2504_13989_b200/synth.py and of the benchmark's tables: d_pad = m * 2^k.
"""
from __future__ import annotations

import math

import torch

from paper_2504_13989_b200 import Plan

DEV = "cuda:0"
DTYPES = {"bf16": torch.bfloat16, "f32": torch.float32}

# (d, d_pad, m): hidden widths, widths of MLP inputs, and the hidden width that is expanded to a full Paley order
HIDDEN = [(4096, 4096, 1), (3584, 3584, 28), (4096, 4096, 1), (3584, 3584, 28), (5120, 5120, 20), (8192, 8192, 1)]
MLP = [(18944, 20480, 20), (14336, 14336, 28), (11008, 11264, 44)]
PALEY = (1536, 1544, 1544)


def _case(name, kind, width, rows, bits, group=0, alpha=0.9, dtype="bf16", **more):
    d, d_pad, m = width
    return {"name": name, "kind": kind, "rows": rows, "d": d, "d_pad": d_pad, "m": m, "bits": bits, "group": group,
            "alpha": alpha, "dtype": dtype, **more}


def listed():
    return [
        # one decoding step of a small batch: 16 tokens' hidden states before a projection
        _case("decode_hidden", "quantize", (4096, 4096, 1), 16, 4),
        # one prefill chunk of hidden states, one scale per token
        _case("prefill_hidden", "quantize", (4096, 4096, 1), 4096, 3),
        # two prompts at the 3584-wide model's hidden size, scales per 128 coordinates
        _case("prefill_grouped", "quantize", (3584, 3584, 28), 8192, 3, 128, 0.85),
        # the input of an MLP's down projection, expanded 18944 -> 20480; a ragged batch of prompts
        _case("prefill_mlp", "quantize", (18944, 20480, 20), 4001, 4, 0, 0.95),
        # KV entries of a whole prompt batch (16 sequences x 32 heads x 4096 tokens), asymmetric as the cache stores them
        _case("kv_write", "quantize", (128, 128, 1), 16 * 32 * 4096, 4, 128, 1.0, asymmetric=True),
        # fp32 activations (a model kept in fp32, or weights before they are cast) of an odd number of tokens
        _case("hidden_f32", "quantize", (4096, 4096, 1), 3001, 4, 0, 0.9, "f32"),
        # the width that only a full Paley order fits: 1536 -> 1544
        _case("hidden_paley", "quantize", PALEY, 4096, 4),
        # a KV cache read back for attention: 8 sequences' keys of 8 heads x 4096 tokens
        _case("kv_read", "dequantize", (128, 128, 1), 8 * 8 * 4096, 4, 128, 1.0, asymmetric=True, inverse=True),
        # stored activations restored for a layer that runs unquantized, scales per 128 coordinates
        _case("restore_grouped", "dequantize", (3584, 3584, 28), 8192, 3, 128, 0.85, inverse=True),
        # one projection of a decoding step: 16 tokens
        _case("linear_decode", "linear", (4096, 4096, 1), 16, 4, n_out=4096),
        # the same projection of a prefill chunk
        _case("linear_prefill", "linear", (4096, 4096, 1), 4096, 4, n_out=4096),
        # calibration: 32 clip ratios over the activations of 16 sequences x 2048 tokens of one layer
        _case("calibrate", "clip", (4096, 4096, 1), 16 * 2048, 3, candidates=32),
    ]


def _log(rng, lo, hi):
    """A whole number between lo and hi, spread over its logarithm; odd and ragged ones among them."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    what = rng.choice(["hidden", "hidden", "mlp", "kv", "f32", "paley", "kv_read", "restore", "restore", "linear", "linear",
                       "clip"])
    bits = rng.choice([3, 4])
    alpha = rng.choice([0.8, 0.85, 0.9, 0.95, 1.0])
    if what == "hidden":
        c = _case("", "quantize", rng.choice(HIDDEN), _log(rng, 1, 16384), bits, rng.choice([0, 128]), alpha)
    elif what == "mlp":
        c = _case("", "quantize", rng.choice(MLP), _log(rng, 1, 4096), bits, rng.choice([0, 128]), alpha)
    elif what == "kv":
        c = _case("", "quantize", (128, 128, 1), _log(rng, 256, 16 * 32 * 4096), bits, 128, 1.0, asymmetric=rng.random() < 0.7)
    elif what == "f32":
        c = _case("", "quantize", rng.choice(HIDDEN), _log(rng, 1, 8192), bits, rng.choice([0, 128]), alpha, "f32")
    elif what == "paley":
        c = _case("", "quantize", PALEY, _log(rng, 1, 8192), bits, 0, alpha)
    elif what == "kv_read":
        dtype = rng.choice(["bf16", "bf16", "f32"])
        c = _case("", "dequantize", (128, 128, 1), _log(rng, 256, (16 if dtype == "bf16" else 8) * 32 * 4096), bits, 128, 1.0, dtype,
                  asymmetric=rng.random() < 0.7, inverse=True)
    elif what == "restore":
        c = _case("", "dequantize", rng.choice(HIDDEN), _log(rng, 1, 16384), bits, rng.choice([0, 128]), alpha,
                  rng.choice(["bf16", "bf16", "f32"]), inverse=rng.random() < 0.7)
    elif what == "linear":
        tokens = _log(rng, 1, 4096)
        c = _case("", "linear", rng.choice([(4096, 4096, 1), (3584, 3584, 28)]), tokens, bits, 0, alpha,
                  n_out=128 * rng.randint(8, min(112, 4096 * 32 // tokens)))
    else:
        k = rng.choice([8, 16, 31, 32])
        c = _case("", "clip", rng.choice(HIDDEN[:4]), _log(rng, 512, 16 * 2048 * 32 // max(k, 32)), bits, rng.choice([0, 128]), alpha,
                  candidates=k)
    del c["name"]
    return c


def _rows(n, d, gen):
    """Heavy-tailed rows with a few outlier channels and a few massive tokens, as hidden states and KV entries have them."""
    def normal():
        return torch.randn((n, d), generator=gen, device=DEV)
    x, chi = normal(), normal().square_()
    for _ in range(2):
        chi.addcmul_(*(2 * [normal()]))
    x.div_(chi.div_(3.0).sqrt_()).mul_(0.5)
    channels = torch.randperm(d, generator=gen, device=DEV)[: max(4, d // 256)]
    x[:, channels] *= 50.0
    tokens = torch.randperm(n, generator=gen, device=DEV)[: n // 100]
    x[tokens] *= 20.0
    return x


def _stored(case, info, gen):
    """Packed codes and scales as a cache holds them: rotated coordinates are near normal, the largest of a group takes the last code."""
    n, bits, groups = case["rows"], info.bits, info.scales_per_row
    asym = bool(info.asymmetric)
    top = 2 ** bits - 1 if asym else 2 ** (bits - 1) - 1
    q = torch.randn((n, info.d_pad), generator=gen, device=DEV).mul_(top / (6.6 if asym else 3.3))
    q = q.add_(top / 2 if asym else 0.0).round_().clamp_(0 if asym else -top, top).to(torch.int32) & (2 ** bits - 1)
    # little-endian bit stream: eight codes fill `bits` bytes
    q = q.reshape(n, info.d_pad // 8, 8) << (bits * torch.arange(8, dtype=torch.int32, device=DEV))
    word = torch.sum(q, dim=2, dtype=torch.int64)
    codes = torch.stack([(word >> (8 * i) & 255).to(torch.uint8) for i in range(bits)], dim=2).reshape(n, -1)
    delta = torch.rand((n, groups), generator=gen, device=DEV).mul_(0.4).add_(0.1)
    scales = torch.stack([delta, delta * (-top / 2)], dim=2).reshape(n, -1) if asym else delta
    return codes, scales.contiguous()


def prepare(case, seed):
    gen = torch.Generator(device=DEV)
    gen.manual_seed(seed)
    kind, n, d = case["kind"], case["rows"], case["d"]
    plan = Plan(d, case["d_pad"], case["m"], case["bits"], case["group"], case["alpha"], asymmetric=case.get("asymmetric", False))
    state = {"kind": kind, "plan": plan}
    if kind == "dequantize":
        state["codes"], state["scales"] = _stored(case, plan.info, gen)
        state["dtype"], state["inverse"] = DTYPES[case["dtype"]], case["inverse"]
        return state
    state["x"] = _rows(n, d, gen).to(DTYPES[case["dtype"]])
    if kind == "linear":
        w = (torch.randn((case["n_out"], d), generator=gen, device=DEV) / math.sqrt(d)).to(torch.bfloat16)
        state["plan_w"] = Plan(d, case["d_pad"], case["m"], case["bits"], 0, 1.0)
        state["codes_w"], state["scales_w"] = state["plan_w"].weight_rotate_quantize(w)
    elif kind == "clip":
        k = case["candidates"]
        state["alphas"] = [0.5 + 0.5 * (i + 1) / k for i in range(k)]
    return state


def run(state):
    kind, plan = state["kind"], state["plan"]
    if kind == "quantize":
        codes, scales, _ = plan.rotate_quantize(state["x"])
        return codes, scales
    if kind == "dequantize":
        return plan.dequantize(state["codes"], state["scales"], inverse=state["inverse"], dtype=state["dtype"])
    if kind == "linear":
        codes, scales, _ = plan.rotate_quantize(state["x"])
        return plan.quantized_matmul(codes, scales, state["plan_w"], state["codes_w"], state["scales_w"], dtype=torch.bfloat16)
    return plan.clip_error(state["x"], state["alphas"])


def work(case):
    n, d, d_pad, m, bits, group = (case[k] for k in ("rows", "d", "d_pad", "m", "bits", "group"))
    elem = 4 if case["dtype"] == "f32" else 2
    scales = (d_pad // group if group else 1) * (2 if case.get("asymmetric") else 1)
    packed = d_pad * bits // 8 + 4 * scales                                          # bytes of one quantized row
    if m == d_pad:
        rotation = 2 * n * m * d                                                     # no fast transform for a full order
    else:
        rotation = n * d_pad * (math.log2(d_pad // m) + (m if m > 1 else 0))         # butterflies, and the mix of the m blocks
    kind = case["kind"]
    if kind == "quantize":
        return {"bytes": n * (d * elem + packed), "flops": rotation}
    if kind == "dequantize":
        return {"bytes": n * (packed + (d if case["inverse"] else d_pad) * elem), "flops": rotation if case["inverse"] else n * d_pad}
    if kind == "linear":
        o = case["n_out"]
        return {"bytes": n * d * elem + o * packed + n * o * 2, "flops": rotation + 2 * n * o * d_pad}
    return {"bytes": n * d * elem + 8 * case["candidates"], "flops": rotation}


def tolerance(case):
    kind = case["kind"]
    if kind == "quantize":
        # scales are maxima of sums of thousands of fp32 terms; a code may fall to either side of a rounding tie
        return {"rel": 1e-5, "max": 1e-4, "differ": 1e-4}
    if kind == "dequantize":
        return {"rel": 4e-3 if case["dtype"] == "bf16" else 1e-5}                    # one rounding; fp32: sums of fp32 terms
    if kind == "linear":
        return {"rel": 4e-3, "max": 0.1}                                             # exact sums, rounded to bf16 once
    return {"rel": 1e-5, "max": 1e-4}                                                # sums of fp32 squares
