"""A forward whose inputs are the output of the forward queued right before it.  The kernels of one forward start while those
of the one before are still draining (programmatic dependent launch); whatever they load early must not be something that
forward is still writing.  The chain queued without a pause has to equal, bit for bit, the same chain with a wait after
every call."""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, d, ksize, dtype
CASES = [(1, 2, 64, 64, 64, 3, "bf16"), (2, 8, 64, 64, 64, 3, "bf16"), (1, 3, 96, 64, 64, 5, "bf16"),
         (1, 2, 65, 65, 32, 3, "bf16"), (8, 8, 50, 75, 32, 5, "bf16"), (8, 12, 14, 14, 64, 3, "bf16"),
         (2, 4, 14, 14, 32, 3, "f32"), (1, 2, 48, 50, 64, 3, "f32"), (2, 3, 40, 40, 48, 3, "f32")]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_output_of_one_forward_is_the_input_of_the_next(case):
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(*case, seed=1500 + sum(case[:6]))
    s = c.shape
    dev = torch.device("cuda:0")
    x, w, b = c.v.to(dev), c.dw_weight.to(dev), c.dw_bias.to(dev)
    bufs = [torch.empty_like(x) for _ in range(3)]
    busy = torch.randn(4096, 4096, device=dev)
    with CastlingAttn(ksize=s.ksize) as attn:
        def chain(wait):
            src = x
            for out in bufs:
                attn.forward(src, src, src, w, b, s.gridH, s.gridW, out=out)
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
        assert attn.device_status() == (0, 0)


@pytest.mark.parametrize("case", [(2, 8, 64, 64, 64, 3, "bf16"), (1, 2, 48, 50, 64, 3, "f32"), (2, 8, 64, 64, 32, 5, "f32")],
                         ids=lambda c: "x".join(map(str, c)))
def test_output_of_a_forward_is_the_input_of_an_apply_pass_on_its_own(case):
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(*case, seed=1550 + sum(case[:6]))
    s = c.shape
    dev = torch.device("cuda:0")
    x, w, b = c.v.to(dev), c.dw_weight.to(dev), c.dw_bias.to(dev)
    buf = torch.empty_like(x)
    busy = torch.randn(4096, 4096, device=dev)
    with CastlingAttn(ksize=s.ksize) as attn:
        state = attn.shard_state(x, x)
        def chain(wait):
            attn.forward(x, x, x, w, b, s.gridH, s.gridW, out=buf)
            if wait:
                torch.cuda.synchronize()
            return attn.shard_apply(buf, buf, w, b, state, s.gridH, s.gridW, 0, 0)
        want = chain(True).clone()
        for _ in range(20):
            buf.zero_()
            torch.cuda.synchronize()
            busy @ busy
            got = chain(False)
            torch.cuda.synchronize()
            assert torch.equal(got, want), "the apply pass read its input before the forward before it had written it"
        assert attn.device_status() == (0, 0)
