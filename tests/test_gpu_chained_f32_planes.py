"""fp32 forwards of short planes, each on the output of the one queued right before it: the one-kernel form, which lets what follows start before it has itself
waited, the two-kernel form, whose second kernel loads Q and V before its own wait, and each after the other.  The chain queued without a pause,
and the chain replayed from a captured graph, have to equal, bit for bit, the same chain with a wait after every call.
"""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, planes of every other call (0: all): clusters, one CTA per plane, more planes than multiprocessors, both in turn
CASES = [(8, 4, 14, 14, 32, 3, 0), (50, 3, 14, 14, 32, 3, 0), (100, 4, 9, 9, 32, 5, 0), (8, 4, 14, 14, 64, 3, 0), (30, 6, 10, 10, 64, 3, 0),
         (8, 4, 14, 14, 32, 3, 8), (50, 3, 14, 14, 32, 3, 6), (8, 4, 10, 10, 64, 5, 4), (40, 2, 64, 1, 32, 3, 0)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_output_of_one_forward_is_the_input_of_the_next(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, d, ks, few = case
    c = workloads.custom_call(B, H, gh, gw, d, ks, "f32", seed=2900 + B + gh + few)
    dev = torch.device("cuda:0")
    x, w, b = c.v.to(dev), c.dw_weight.to(dev), c.dw_bias.to(dev)
    n = few // H if few else B   # images of every other call
    bufs = [torch.empty_like(x) for _ in range(5)]
    busy = torch.randn(4096, 4096, device=dev)
    with CastlingAttn(ksize=ks) as attn:
        def chain(wait):
            src = x
            for i, out in enumerate(bufs):
                m = n if i % 2 else B
                if m < B:
                    out[m:].copy_(src[m:])
                attn.forward(src[:m], src[:m], src[:m], w, b, gh, gw, out=out[:m])
                if wait:
                    torch.cuda.synchronize()
                src = out
            return src
        want = chain(True).clone()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            chain(False)
        for i in range(20):
            for t in bufs:
                t.zero_()
            torch.cuda.synchronize()
            busy @ busy            # keeps the device busy until the whole chain is queued
            if i % 2:
                graph.replay()
            else:
                chain(False)
            torch.cuda.synchronize()
            assert torch.equal(bufs[-1], want), "a forward read its input before the forward before it had written it"
        assert attn.device_status() == (0, 0)
        del graph
