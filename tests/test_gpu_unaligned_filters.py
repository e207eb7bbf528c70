"""Filters and bias are asked for element alignment only (q, k, v and out for 16 bytes): contiguous ones that begin at an odd
element of their storage, as slices of one flat parameter buffer do, give the same bits as aligned ones on every kernel family
and variant."""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, dtype, kernel family
CASES = [(2, 3, 14, 14, 64, 3, "bf16", 2), (2, 3, 14, 14, 32, 5, "bf16", 2),       # one launch
         (2, 3, 20, 24, 64, 5, "bf16", 2), (2, 3, 24, 24, 32, 3, "bf16", 2),       # state and apply
         (3, 8, 31, 33, 32, 5, "bf16", 2),                                         # ... an odd grid
         (2, 3, 9, 9, 48, 3, "bf16", 1), (40, 4, 5, 5, 32, 3, "bf16", 1),          # CUDA cores
         (2, 3, 20, 24, 64, 3, "f32", 1), (2, 3, 9, 9, 48, 7, "f32", 1)]
VARIANTS = [{}, {"normalize_rows": True}, {"exact_kernel": True}, {"sparse_eps": 0.01}]


def odd_view(t):
    flat = torch.empty(t.numel() + 1, dtype=t.dtype, device=t.device)
    view = flat[1:].view_as(t)
    view.copy_(t)
    assert view.is_contiguous() and view.data_ptr() % (2 * t.element_size()) == t.element_size()
    return view


@pytest.mark.parametrize("variant", VARIANTS, ids=lambda v: next(iter(v), "core"))
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_filters_and_bias_at_an_odd_element(case, variant):
    from paper_2211_10526_b200 import CastlingAttn
    *shape, family = case
    c = workloads.custom_call(*shape, seed=1700 + sum(shape[:6]))
    s = c.shape
    dev = torch.device("cuda:0")
    q, k, v, w, b = (t.to(dev) for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    with CastlingAttn(ksize=s.ksize, **variant) as attn:
        want = attn.forward(q, k, v, w, b, s.gridH, s.gridW)
        if not ({"exact_kernel", "sparse_eps"} & set(variant)) or s.d == 64:
            assert attn.last_path()[0] == family
        got = attn.forward(q, k, v, odd_view(w), odd_view(b), s.gridH, s.gridW)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    assert torch.equal(got, want)
