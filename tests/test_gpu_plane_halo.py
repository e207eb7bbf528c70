"""Single-kernel forward on both sides of the line between planes that fit its buffers with the convolution's halo and those that do
not: the last grid that fits and the first that does not, rows and columns of one token, leading tokens, both CTA shapes, both
widths, both filter sizes, against the float64 oracle.
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
CASES = [(2, 3, 14, 14, 64, 3, "heads", 16), (2, 3, 14, 15, 64, 3, "heads", 0), (2, 3, 1, 83, 64, 3, "tokens", 0),
         (2, 3, 1, 84, 64, 3, "heads", 1), (2, 3, 83, 1, 64, 3, "heads", 0), (2, 3, 84, 1, 64, 3, "fused", 0),
         (2, 3, 12, 12, 64, 5, "fused", 1), (2, 3, 12, 13, 64, 5, "heads", 0), (2, 3, 16, 16, 64, 3, "heads", 0),
         (160, 3, 6, 14, 64, 3, "heads", 2), (160, 3, 7, 13, 64, 3, "heads", 0),
         (3, 4, 21, 20, 32, 3, "heads", 4), (3, 4, 22, 22, 32, 3, "heads", 0), (3, 4, 1, 168, 32, 3, "heads", 0),
         (3, 4, 2, 126, 32, 3, "tokens", 0), (3, 5, 13, 11, 32, 5, "heads", 0), (80, 4, 9, 11, 32, 3, "heads", 1)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_halo_in_the_plane_buffer(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, layout, prefix = case
    dev = torch.device("cuda:0")
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "bf16", seed=2100 + gh + gw, qk_lognormal_sigma=0.5)
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
