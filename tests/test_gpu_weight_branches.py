"""Exact angular kernel on the tensor cores where its weight function takes its two forms, against the float64 oracle: a step of
cosines that are all small takes one, a step that holds a large one the other.  Planes whose keys are turned towards the queries so
that cosines lie on both sides of the line, at it, and at 1 and -1; sizes with full and ragged tiles.

Bound: a cosine of unit rows rounded to bf16 is off by at most 2^-8, which moves a weight 1 - arccos(x)/pi by the larger of
its two neighbours' distances; the weight and the output are rounded to bf16 (2^-9 each); 1e-4 covers the approximation of
arccos.  An output is off by at most the sum of that over the keys times |v|, and by its own rounding.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


def cosines(q, k):
    q, k = q.double().numpy(), k.double().numpy()
    return np.clip((q / np.linalg.norm(q, axis=-1, keepdims=True)) @ (k / np.linalg.norm(k, axis=-1, keepdims=True)).T, -1, 1)


@pytest.mark.parametrize("mix", [0.55, 0.6, 0.65, 0.95, 1.0, -0.6, -1.0])
@pytest.mark.parametrize("grid", [(1, 16), (5, 13), (16, 16), (3, 43)], ids=lambda g: f"{g[0]}x{g[1]}")
def test_small_and_large_cosines(grid, mix):
    from paper_2211_10526_b200 import CastlingAttn
    gh, gw = grid
    c = workloads.custom_call(1, 2, gh, gw, 64, 3, "bf16", seed=77)
    # every third key of head 0, and every key of head 1 around one direction, at the cosine `mix` of a query
    q, k = c.q.float(), c.k.float()
    unit = lambda t: t / t.norm(dim=-1, keepdim=True)
    k[:, 0, ::3] = mix * unit(q[:, 0, ::3]) + (1 - mix * mix) ** 0.5 * unit(k[:, 0, ::3])
    k[:, 1] = mix * unit(q[:, 1, :1]) + (1 - mix * mix) ** 0.5 * unit(k[:, 1])
    k = k.to(torch.bfloat16)
    dev = torch.device("cuda:0")
    with CastlingAttn(ksize=3, exact_kernel=True, force_path=2) as attn:
        out = attn.forward(c.q.to(dev), k.to(dev), c.v.to(dev), c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    got = out.double().cpu().numpy()
    ref = oracle.forward_matrix(c.q, k, c.v, c.dw_weight, c.dw_bias, gh, gw, 3, threads=8, kernel=oracle.KERNEL_EXACT)
    for h in range(2):
        x = cosines(c.q[0, h], k[0, h])
        w = lambda y: 1 - np.arccos(np.clip(y, -1, 1)) / np.pi
        dw = np.maximum(w(x + 2.0 ** -8) - w(x), w(x) - w(x - 2.0 ** -8)) + 2.0 ** -9 * w(x) + 1e-4 / np.pi
        bound = dw @ np.abs(c.v[0, h].double().numpy()) + 2.0 ** -9 * np.abs(ref[0, h]) + 1e-6
        err = np.abs(got[0, h] - ref[0, h])
        assert np.all(err <= bound), f"head {h}: largest error over its bound: {float(np.max(err / bound)):.2f}"
