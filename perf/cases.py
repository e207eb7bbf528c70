"""The work a user of the attention core has it do: cases to time and compare, through ``CastlingAttn.forward``.

A case is one call of the core: ``B`` images, ``H`` heads of width ``d``, ``prefix`` leading off-grid tokens and a
``gridH x gridW`` token grid, a ``ksize x ksize`` depthwise filter, the element type, the memory layout of the four
token tensors and the variant of the attention:

* layout ``heads``: contiguous ``[B, H, N, d]``; ``tokens``: token-major ``[B, N, H, d]``, what a projection layer
  leaves; ``fused``: q, k and v are slices of one ``[B, N, 3, H, d]`` projection (the output is token-major);
* variant ``core`` (the inference-time attention), ``rownorm`` (rows of weights divided by their sums), ``exact``
  (the exact angular kernel), ``masked`` (the core plus the masked softmax branch of training).

Values are Gaussian; ``scale`` > 0 multiplies every row of q and k by a log-normal factor with that sigma, as the
rows of trained projections differ in length.  Filters and bias have the standard deviation 0.1.
"""
from __future__ import annotations

import math

import torch

from paper_2211_10526_b200 import CastlingAttn

_DTYPES = {"f32": torch.float32, "bf16": torch.bfloat16}
_BYTES = {"f32": 4, "bf16": 2}


def _case(B, H, gridH, gridW, d, ksize, dtype, layout="heads", prefix=0, variant="core", scale=0.0):
    return {"B": B, "H": H, "gridH": gridH, "gridW": gridW, "d": d, "ksize": ksize, "dtype": dtype,
            "layout": layout, "prefix": prefix, "variant": variant, "scale": scale}


def listed():
    cases = {
        # the fp32 check configuration: a call whose time is launches and host work
        "fp32_tiny": _case(2, 4, 14, 14, 32, 3, "f32"),
        # one image through a DeiT-Base-shaped layer (class token, fused projection): latency of online inference
        "one_image": _case(1, 12, 14, 14, 64, 3, "bf16", "fused", prefix=1, scale=0.5),
        # the first and second stage of a LeViT-shaped network on a batch of 64; the second has an odd grid
        "levit_14x14": _case(64, 4, 14, 14, 32, 3, "bf16"),
        "levit_7x7": _case(64, 8, 7, 7, 32, 3, "bf16"),
        # a DeiT-Base-shaped layer on a batch of 64: throughput of classification
        "deit_batch": _case(64, 12, 14, 14, 64, 3, "bf16", "fused", prefix=1, scale=0.5),
        # a detection backbone at high resolution with 5x5 filters: square input, and a photograph of 800 x 1200
        # pixels at a stride of 16
        "detection_64x64": _case(8, 8, 64, 64, 32, 5, "bf16"),
        "detection_50x75": _case(8, 8, 50, 75, 32, 5, "bf16"),
        # the long-sequence sweep: a middle point, with the rows of weights normalised, and the largest one
        "rownorm_128x128": _case(2, 8, 128, 128, 64, 3, "bf16", variant="rownorm"),
        "sweep_256x256": _case(2, 8, 256, 256, 64, 3, "bf16"),
        # evaluation in full precision on a long sequence
        "fp32_128x128": _case(2, 8, 128, 128, 64, 3, "f32"),
        # explicit weights: the exact angular kernel that the kept one is compared with, and a training-time forward
        # with the masked softmax branch
        "exact_64x64": _case(2, 8, 64, 64, 64, 3, "bf16", variant="exact"),
        "masked_deit": _case(64, 12, 14, 14, 64, 3, "bf16", variant="masked", scale=0.5),
    }
    return [dict(c, name=n) for n, c in cases.items()]


def _log(rng, lo, hi):
    """An integer of [lo, hi], uniform in its logarithm."""
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case: the kinds of work above over the whole range of batch, heads and grid sides."""
    kind = rng.choice(["core", "core", "core", "rownorm", "f32", "exact", "masked"])
    d = rng.choice([32, 64])
    heads = rng.choice([3, 4, 6, 8, 12, 16])
    ksize = rng.choice([3, 3, 3, 5])
    layout = rng.choice(["heads", "heads", "tokens", "fused"])
    scale = rng.choice([0.0, 0.5])
    while True:
        batch = _log(rng, 1, 64)
        quadratic = kind in ("exact", "masked")
        side = 28 if kind == "masked" else 64 if kind == "exact" else 256
        gridH = _log(rng, 4, side)
        gridW = gridH if rng.random() < 0.4 else _log(rng, 4, side)
        N = gridH * gridW
        planes = batch * heads
        if quadratic:
            fits = planes * N * N <= (2 * 8 * 4096 ** 2 if d == 64 else 1 << 24)
        elif kind == "core" and d == 64:
            fits = planes * N <= 2 * 8 * 256 ** 2
        else:
            fits = planes * N <= 2 * 8 * 128 ** 2
        if fits:
            break
    prefix = rng.choice([0, 1, 2]) if kind in ("core", "rownorm", "f32") and N <= 1024 else 0
    return _case(batch, heads, gridH, gridW, d, ksize, "f32" if kind == "f32" else "bf16", layout, prefix,
                 "core" if kind == "f32" else kind, scale)


def prepare(case, seed):
    """The tensors a layer has in hand before the call, drawn on the GPU, and the handle it keeps."""
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev)
    gen.manual_seed(seed)
    B, H, d, ks, prefix = case["B"], case["H"], case["d"], case["ksize"], case["prefix"]
    N = prefix + case["gridH"] * case["gridW"]
    dt = _DTYPES[case["dtype"]]

    def rows(scaled):
        t = torch.randn(B, H, N, d, generator=gen, device=dev)
        if scaled and case["scale"] > 0:
            t *= torch.exp(case["scale"] * torch.randn(B, H, N, 1, generator=gen, device=dev))
        return t.to(dt)

    q, k, v = rows(True), rows(True), rows(False)
    if case["layout"] == "fused":
        qkv = torch.stack([t.permute(0, 2, 1, 3) for t in (q, k, v)], dim=2)  # [B, N, 3, H, d]
        q, k, v = (qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3))
    elif case["layout"] == "tokens":
        q, k, v = (t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v))
    w = (0.1 * torch.randn(H * d, ks, ks, generator=gen, device=dev)).to(dt)
    b = (0.1 * torch.randn(H * d, generator=gen, device=dev)).to(dt)
    variant = case["variant"]
    # the mask's threshold is a little above the mean probability: a few percent of the pairs pass
    attn = CastlingAttn(ksize=ks, prefix_tokens=prefix, normalize_rows=variant == "rownorm",
                        exact_kernel=variant == "exact", sparse_eps=1.25 / N if variant == "masked" else None)
    return {"attn": attn, "args": (q, k, v, w, b, case["gridH"], case["gridW"])}


def run(state):
    """One call of the core, as a layer's forward makes it; the output is a new tensor."""
    return state["attn"].forward(*state["args"])


def work(case):
    """Q, K, V and the filters read once and the output written once; the contractions and the convolution."""
    planes, grid, d = case["B"] * case["H"], case["gridH"] * case["gridW"], case["d"]
    N = case["prefix"] + grid
    e = _BYTES[case["dtype"]]
    taps = case["ksize"] ** 2
    pairs = N * N if case["variant"] in ("exact", "masked") else N * d
    return {"bytes": 4 * planes * N * d * e + case["H"] * d * (taps + 1) * e,
            "flops": planes * (4 * pairs * d + 2 * taps * grid * d)}


def tolerance(case):
    """About four times what the path differs from the same attention in 64 bits, the largest over the listed cases and
    36 drawn ones: fp32 5.3e-7 (largest element 2.6e-6); bf16 1.7e-3 (5.0e-3), and 2.5e-3 (1.2e-2) where the explicit
    weights are rounded to bf16 between the two contractions."""
    if case["dtype"] == "f32":
        return {"rel": 2.5e-6, "max": 1.2e-5}
    if case["variant"] in ("exact", "masked"):
        return {"rel": 1e-2, "max": 5e-2}
    return {"rel": 7e-3, "max": 2e-2}
