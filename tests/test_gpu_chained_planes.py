"""Forwards of short planes and with explicit weights, each on the output of the one queued right before it: their kernels start while
that one drains and wait for it before they touch memory.  The chain queued without a pause has to equal, bit for bit, the same
chain with a wait after every call."""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, variant: one plane per CTA and several, both widths, a forward of two kernels in between
CASES = [(1, 12, 14, 14, 64, 3, {}), (64, 12, 14, 14, 64, 3, {}), (8, 8, 7, 7, 32, 3, {}), (64, 16, 16, 16, 32, 3, {}),
         (2, 8, 24, 24, 64, 3, {"exact_kernel": True}), (64, 4, 14, 14, 64, 3, {"sparse_eps": 1.25 / 196}),
         (8, 12, 14, 14, 64, 3, {"normalize_rows": True})]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:6])) + "".join(c[6]))
def test_output_of_one_forward_is_the_input_of_the_next(case):
    from paper_2211_10526_b200 import CastlingAttn
    *shape, variant = case
    c = workloads.custom_call(*shape, "bf16", seed=1600 + sum(shape))
    s = c.shape
    dev = torch.device("cuda:0")
    x, w, b = c.v.to(dev), c.dw_weight.to(dev), c.dw_bias.to(dev)
    bufs = [torch.empty_like(x) for _ in range(4)]
    busy = torch.randn(4096, 4096, device=dev)
    with CastlingAttn(ksize=s.ksize, **variant) as attn, CastlingAttn(ksize=s.ksize) as other:
        def chain(wait):
            src = x
            for i, out in enumerate(bufs):
                (other if i == 2 else attn).forward(src, src, src, w, b, s.gridH, s.gridW, out=out)
                if wait:
                    torch.cuda.synchronize()
                src = out
            return src
        want = chain(True).clone()
        for _ in range(20):
            for t in bufs:
                t.zero_()
            torch.cuda.synchronize()
            busy @ busy            # keeps the device busy until the whole chain is queued
            got = chain(False)
            torch.cuda.synchronize()
            assert torch.equal(got, want), "a forward read its input before the forward before it had written it"
        assert attn.device_status() == (0, 0) and other.device_status() == (0, 0)
