"""Width-32 heads in 64-byte rows on the tensor-core kernels (odd grid widths, odd token counts, an odd number of heads side
by side), against the float64 oracle at the edges of their tiles: 256-token stages of the state kernel with one token less
or more, patches of 8 x 32 and 16 x 16 tokens with a row or a column less or more, one column, several token splits, leading tokens, both
filter sizes, the row-sum division; and each term of Eq. 9 on its own scale.  Bound: 2e-2 of the largest output, as for
every bf16 shape (output rounding 2^-9, operands rounded to bf16).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, ksize, layout, prefix
CASES = [(4, 5, 15, 17, 3, "heads", 0), (4, 5, 1, 257, 3, "heads", 0), (3, 6, 7, 33, 5, "heads", 0),
         (3, 6, 9, 31, 3, "heads", 0), (20, 3, 73, 1, 3, "heads", 0), (1, 2, 90, 57, 5, "heads", 0),
         (8, 3, 16, 16, 3, "tokens", 0), (4, 5, 8, 32, 5, "fused", 0), (3, 3, 24, 40, 3, "heads", 1),
         (5, 3, 17, 31, 5, "tokens", 2), (60, 8, 7, 7, 3, "heads", 0),
         (8, 9, 17, 15, 3, "heads", 0), (8, 9, 32, 17, 5, "tokens", 1), (8, 8, 31, 33, 5, "heads", 0), (8, 9, 33, 16, 3, "fused", 0)]


def views(c, layout, dev):
    if layout == "heads":
        q, k, v = (t.to(dev) for t in (c.q, c.k, c.v))
        return q, k, v, torch.full_like(q, float("nan"))
    s = c.shape
    out = torch.full((s.B, s.N, s.H, s.d), float("nan"), dtype=c.q.dtype, device=dev).permute(0, 2, 1, 3)
    if layout == "tokens":
        return (*(t.permute(0, 2, 1, 3).contiguous().to(dev).permute(0, 2, 1, 3) for t in (c.q, c.k, c.v)), out)
    qkv = torch.stack([t.permute(0, 2, 1, 3) for t in (c.q, c.k, c.v)], dim=2).to(dev)
    return (*(qkv[:, :, i].permute(0, 2, 1, 3) for i in range(3)), out)


def run(c, gh, gw, layout, prefix, rownorm, what):
    from paper_2211_10526_b200 import CastlingAttn
    dev = torch.device("cuda:0")
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=c.shape.ksize, prefix_tokens=prefix, normalize_rows=rownorm) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path()[0] == 2
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, c.shape.ksize,
                                                                  threads=8, prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))
    assert err <= 2e-2, f"{what}: max-rel error {err:.3e}"


@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_tile_edges(case, rownorm):
    B, H, gh, gw, ks, layout, prefix = case
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, 32, ks, "bf16", seed=1200 + gh + gw, qk_lognormal_sigma=0.5)
    run(c, gh, gw, layout, prefix, rownorm, "all terms")


@pytest.mark.parametrize("ks", [3, 5])
@pytest.mark.parametrize("term", ["conv", "linear", "halfsum"])
def test_one_term_at_a_time(term, ks):
    gh, gw = 33, 43
    c = workloads.custom_call(3, 5, gh, gw, 32, ks, "bf16", seed=1300 + ks)
    if term != "halfsum":   # antisymmetric along the tokens: the token sum is exactly zero
        n = gh * gw // 2
        c.v[:, :, n + 1:] = -c.v[:, :, :n].flip(2)
        c.v[:, :, n] = 0
    if term == "conv":
        c.dw_weight = (c.dw_weight.float() * 30).to(c.dw_weight.dtype)
        c.dw_bias = (c.dw_bias.float() * 20).to(c.dw_bias.dtype)
    else:
        c.dw_weight.zero_(); c.dw_bias.zero_()
    if term != "linear":
        c.k.zero_()
    run(c, gh, gw, "heads", 0, False, term)
