"""Single-kernel forward: each tap of the convolution at the edges of the grid, on its own scale.  K is zero, and so is the sum of V over the tokens, V and -V
in pairs of tokens, so that the output is the convolution alone and its rounding to bf16 the only error; filters have the size of V.  A tap that
read a token across an edge instead of zero, or missed one, would be off by a whole product of that size.

Bound, element by element: 2^-8 of the value for the rounding (2^-9) and fp32 sums of 25 products of bf16 (25 * 2^-23 of their sum of magnitudes).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_narrow_rows import views
from test_gpu_plane_halo import CASES as HALO_CASES

pytestmark = pytest.mark.gpu

CASES = HALO_CASES + [(2, 3, 1, 100, 64, 5, "fused", 2), (2, 3, 1, 256, 64, 3, "heads", 0), (160, 2, 1, 60, 64, 5, "tokens", 0)]   # rows taken as columns


def inputs(case):
    B, H, gh, gw, d, ks, layout, prefix = case
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "bf16", seed=3100 + gh + gw, w_std=1.0)
    N = prefix + gh * gw
    order = torch.randperm(N, generator=torch.Generator().manual_seed(7))
    c.k.zero_()
    c.v[:, :, order[N // 2:2 * (N // 2)]] = -c.v[:, :, order[:N // 2]]
    if N % 2:
        c.v[:, :, order[-1]] = 0
    return c


def bound(c, gh, gw, ks, prefix, ref):
    most = oracle.forward(c.q, c.k, c.v.abs(), c.dw_weight.abs(), c.dw_bias.abs(), gh, gw, ks, threads=8, prefix=prefix)   # sums of magnitudes, the token sum's among them
    return 2.0 ** -8 * np.abs(ref) + 25 * 2.0 ** -23 * most + 1e-6


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_every_tap(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, layout, prefix = case
    dev = torch.device("cuda:0")
    c = inputs(case)
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=ks, prefix_tokens=prefix, force_path=2) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path() == (2, 1)
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = np.abs(got - ref) / bound(c, gh, gw, ks, prefix, ref)
    assert np.all(err <= 1), f"largest error over its bound: {float(err.max()):.2f}"
