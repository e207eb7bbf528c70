"""fp32 forward of short planes, in one kernel or (a few planes) two, at the edges of its splits, against the float64 oracle: one, two and four CTAs per plane with
bands of unequal height, rows and columns of one token, the most tokens it takes, leading tokens, several planes per
multiprocessor, strided layouts.  Bound: sums of at most 256 fp32 terms, error about sqrt(N) 2^-24 of the largest partial sum; 1e-5 of
the largest output covers it (measured below 2e-6).
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
CASES = [(1, 1, 1, 1, 32, 3, "heads", 0), (2, 4, 14, 14, 32, 3, "heads", 0), (2, 4, 14, 14, 64, 5, "fused", 1), (1, 3, 15, 16, 32, 3, "tokens", 16),
         (1, 2, 5, 51, 32, 5, "heads", 0), (1, 1, 256, 1, 32, 3, "heads", 0), (1, 2, 1, 254, 32, 3, "heads", 1), (1, 2, 1, 60, 64, 5, "heads", 0),
         (2, 3, 2, 100, 64, 3, "heads", 0), (3, 5, 11, 8, 64, 3, "tokens", 2), (40, 5, 7, 7, 32, 5, "heads", 0), (5, 4, 14, 15, 32, 3, "tokens", 1), (6, 4, 12, 12, 64, 3, "heads", 0), (150, 1, 13, 17, 32, 3, "heads", 3),
         (30, 5, 10, 10, 64, 3, "heads", 0), (37, 4, 14, 14, 64, 3, "fused", 0), (37, 2, 9, 9, 32, 3, "heads", 0)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_bands_of_a_plane(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, layout, prefix = case
    dev = torch.device("cuda:0")
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "f32", seed=2300 + gh + gw, qk_lognormal_sigma=0.5)
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=ks, prefix_tokens=prefix) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path() == (1, 1 if B * H >= 20 else 2)
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))
    assert err <= 1e-5, f"max-rel error {err:.3e}"
