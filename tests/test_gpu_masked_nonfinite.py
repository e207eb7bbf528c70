"""Masked branch on the tensor cores with rows that hold a NaN or an infinity: what has no value is NaN, and nothing else is touched.  A query row without a
direction takes its own output row, a key row every output row of its plane (each one's probabilities have it in their sum); other planes stay, bit for bit.
"""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")], ids=str)
@pytest.mark.parametrize("grid", [(7, 7), (14, 14), (20, 30)], ids=lambda g: f"{g[0]}x{g[1]}")
def test_rows_without_a_direction(grid, value):
    from paper_2211_10526_b200 import CastlingAttn
    gh, gw = grid
    N = gh * gw
    c = workloads.custom_call(2, 3, gh, gw, 64, 3, "bf16", seed=3300 + N)
    q, k, v, w, b = (t.cuda() for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    with CastlingAttn(ksize=3, sparse_eps=1.25 / N, force_path=2) as attn:
        want = attn.forward(q, k, v, w, b, gh, gw)
        q[0, 1, N - 1, 5] = value
        k[1, 2, N // 2, 60] = value
        got = attn.forward(q, k, v, w, b, gh, gw)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    nan = torch.zeros_like(got, dtype=torch.bool)
    nan[0, 1, N - 1] = nan[1, 2] = True
    assert torch.equal(torch.isnan(got), nan)
    assert torch.equal(got[~nan], want[~nan])
