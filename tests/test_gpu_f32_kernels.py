"""The fp32 kernels for head widths 32, 64 and 128 at the edges of their tiles, against the float64 oracle: 64-token tiles of
the state kernel with a token less or more, one to many token splits (up to four are added by the apply kernel, more by a
kernel in between), patches of 8 rows x 8, 16 or 32 columns with a row or a column less or more (up to several per CTA, across
planes), leading tokens in a patch of their own, strided layouts, the row-sum division.  Bound: sums of at most N <= 8 192 fp32 terms in blocks, error about
sqrt(N) 2^-24 of the largest partial sum, 1e-5 of the largest output covers it (measured below 2e-6).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, ksize, layout, prefix
CASES = [(1, 1, 1, 1, 3, "heads", 0), (2, 3, 7, 9, 5, "heads", 0), (2, 3, 1, 65, 3, "heads", 0), (1, 2, 8, 32, 5, "tokens", 0),
         (1, 3, 9, 33, 3, "heads", 1), (2, 2, 17, 15, 3, "tokens", 2), (1, 1, 70, 117, 3, "heads", 0), (40, 5, 16, 17, 5, "heads", 0),
         (1, 2, 3, 31, 3, "heads", 16), (31, 5, 25, 33, 3, "tokens", 2), (26, 4, 9, 9, 5, "heads", 1)]


@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("d", [32, 64, 128])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_tile_edges(case, d, rownorm):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, ks, layout, prefix = case
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "f32", seed=1600 + gh + gw + d, qk_lognormal_sigma=0.5)
    dev = torch.device("cuda:0")
    q, k, v = (t.to(dev) for t in (c.q, c.k, c.v))
    out = torch.full_like(q, float("nan"))
    if layout == "tokens":
        q, k, v, out = (t.permute(0, 2, 1, 3).contiguous().permute(0, 2, 1, 3) for t in (q, k, v, out))
    with CastlingAttn(ksize=ks, prefix_tokens=prefix, normalize_rows=rownorm) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8,
                                                                  prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))
    assert err <= 1e-5, f"max-rel error {err:.3e}"
