"""The bound that holds the convolution at the grid's edges rejects what it is there for: one tap that meets a token across the edge instead of
zero, planted in the oracle's output.
"""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import test_gpu_halo_taps as taps

CASES = [c for c in taps.CASES if c[0] <= 3 and min(c[2], c[3]) > 1]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_a_wrong_tap_is_far_outside(case):
    B, H, gh, gw, d, ks, layout, prefix = case
    c = taps.inputs(case)
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, prefix=prefix)
    bound = taps.bound(c, gh, gw, ks, prefix, ref)
    # the upper right tap next to the centre of token (1, gw - 1), beyond the edge, meets token (1, 0), which follows (0, gw - 1) in memory
    v, w = c.v.float().numpy(), c.dw_weight.float().numpy().reshape(H, d, ks, ks)
    r = ks // 2
    wrong = ref.copy()
    wrong[:, :, prefix + gw + gw - 1] += w[None, :, :, r - 1, r + 1] * v[:, :, prefix + gw]
    rejected = np.abs(wrong - ref) > bound
    assert np.mean(rejected[:, :, prefix + 2 * gw - 1]) > 0.9, "one wrong corner tap would pass"
    assert np.all(np.any(rejected, axis=(2, 3)))
