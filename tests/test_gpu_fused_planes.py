"""Single-kernel forward on both of its CTA shapes, against the float64 oracle where it can go wrong: planes one token below,
at and above 128 (and 256) lines, few planes (256 workers) and more than are in flight (128 workers, several planes per
CTA), odd token counts of width 32, strips and segments that leave a remainder, leading tokens, strided layouts.
Bound: 2e-2 of the largest output, as for every bf16 shape (output rounding 2^-9, operands rounded to bf16).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_narrow_rows import views

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, layout, prefix
CASES = [(2, 3, 1, 127, 64, 3, "heads", 0), (2, 3, 16, 8, 64, 5, "tokens", 0), (2, 3, 43, 3, 64, 3, "heads", 0),
         (2, 3, 15, 17, 64, 3, "heads", 1), (160, 2, 9, 14, 64, 3, "heads", 2), (160, 2, 11, 11, 64, 5, "fused", 0),
         (320, 1, 1, 48, 64, 3, "heads", 0), (160, 2, 43, 3, 64, 3, "heads", 0),
         (6, 4, 5, 51, 32, 3, "heads", 0), (3, 4, 64, 4, 32, 5, "tokens", 0), (5, 4, 257, 1, 32, 3, "heads", 1),
         (2, 5, 7, 73, 32, 3, "heads", 1), (4, 5, 7, 37, 32, 5, "heads", 0), (80, 4, 7, 7, 32, 3, "heads", 0),
         (160, 4, 15, 17, 32, 3, "heads", 0), (80, 4, 3, 85, 32, 5, "fused", 1), (80, 4, 2, 128, 32, 3, "heads", 0),
         (160, 4, 3, 86, 32, 3, "heads", 0), (450, 1, 11, 11, 64, 3, "heads", 0)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_plane_edges(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, layout, prefix = case
    dev = torch.device("cuda:0")
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "bf16", seed=1700 + gh + gw, qk_lognormal_sigma=0.5)
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=ks, prefix_tokens=prefix, force_path=2) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path() == (2, 1)
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))
    assert err <= 2e-2, f"max-rel error {err:.3e}"
