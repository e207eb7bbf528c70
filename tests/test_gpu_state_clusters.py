"""Token splits of the state kernel that meet in a cluster, against the float64 oracle and bit for bit against themselves: every number of
splits from two to eight, last splits that are short, and the calls beside them whose splits meet in memory (more planes than leave
each CTA a multiprocessor, more tokens than eight splits take); both widths, operand pairs, the row-sum division.
Bound: 2e-2 of the largest output, as for every bf16 shape (output rounding 2^-9, operands rounded to bf16).
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, rownorm
CASES = [(1, 2, 9, 15, 64, 3, True), (1, 1, 16, 24, 64, 3, False), (1, 1, 17, 37, 64, 5, False), (1, 1, 22, 32, 64, 3, True), (1, 1, 28, 31, 64, 3, False),
         (2, 8, 31, 33, 64, 3, False), (1, 3, 33, 33, 64, 3, True), (3, 6, 32, 32, 64, 3, False), (19, 1, 32, 32, 64, 3, False), (1, 1, 129, 127, 64, 3, False),
         (1, 1, 130, 128, 64, 3, False), (37, 2, 20, 30, 64, 3, False), (2, 4, 48, 64, 32, 3, False), (2, 3, 33, 41, 32, 5, True), (1, 2, 65, 63, 32, 3, False),
         (49, 2, 24, 24, 32, 3, False)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_splits(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, rownorm = case
    dev = torch.device("cuda:0")
    c = workloads.custom_call(B, H, gh, gw, d, ks, "bf16", seed=2500 + gh + gw, qk_lognormal_sigma=0.5)
    q, k, v, w, b = (t.to(dev) for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    with CastlingAttn(ksize=ks, normalize_rows=rownorm, force_path=2) as attn:
        out = attn.forward(q, k, v, w, b, gh, gw)
        again = [attn.forward(q, k, v, w, b, gh, gw) for _ in range(8)]
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path() == (2, 2)
    assert all(torch.equal(out, x) for x in again), "the same call gave another result"
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8)
    err = float(np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref)))
    assert err <= 2e-2, f"max-rel error {err:.3e}"
