"""Explicit-weights attention on the tensor cores at the edges of its tiling, against the float64 oracle: planes of one
token, one token beside a tile of 128 keys or a half or quarter of it, two and three key tiles (the masked branch keeps
two in shared memory between its sweeps), one or two query tiles per work item with a last item of one tile, several
items per multiprocessor.

Bound: weights, unit rows and the output are rounded to bf16 (2^-9 each) and a row of the output is a sum of weights of
one sign times values, so an element is off by at most 4 * 2^-9 of the sum of |w v|; 2e-2 of the largest output covers that.
A cosine of rounded unit rows is off by at most 2^-8, a probability by twice that relatively: a pair that close to the
mask's threshold may fall on either side, which moves an output of its query by that probability times |v|.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, ksize
CASES = [(1, 2, 1, 1, 3), (2, 3, 1, 16, 3), (2, 3, 3, 11, 5), (2, 3, 5, 13, 3), (2, 3, 1, 127, 3), (2, 3, 8, 16, 5),
         (2, 3, 3, 43, 3), (40, 8, 3, 43, 3), (20, 3, 1, 257, 3), (2, 3, 16, 16, 5), (1, 3, 19, 21, 3)]


@pytest.mark.parametrize("variant", ["exact", "masked", "both"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_tile_edges(case, variant):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, ks = case
    c = workloads.custom_call(B, H, gh, gw, 64, ks, "bf16", seed=900 + sum(case))
    exact, thr = variant != "masked", None if variant == "exact" else 1.1 / (gh * gw)
    ref = oracle.forward_matrix(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, sparse_eps=thr,
                                kernel=oracle.KERNEL_EXACT if exact else oracle.KERNEL_LINEAR)
    dev = torch.device("cuda:0")
    q, k, v, w, b = (t.to(dev) for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    out = torch.full_like(q, float("nan"))
    with CastlingAttn(ksize=ks, exact_kernel=exact, sparse_eps=thr, force_path=2) as attn:
        attn.forward(q, k, v, w, b, gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    bound = 2e-2 * np.max(np.abs(ref), axis=(2, 3))  # per plane
    if thr is not None:
        for i in range(B * H):
            b_, h_ = divmod(i, H)
            p = oracle.softmax_probs(c.q[b_, h_], c.k[b_, h_])
            close = np.where(np.abs(p / thr - 1.0) <= 2.0 * 2.0 ** -8, p, 0.0).sum(axis=1).max()
            bound[b_, h_] += close * float(c.v[b_, h_].float().abs().max())
    err = np.max(np.abs(got - ref), axis=(2, 3))
    assert np.all(err <= bound), f"largest error over its bound: {float(np.max(err / bound)):.2f}"
