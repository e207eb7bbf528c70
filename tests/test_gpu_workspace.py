"""The handle's workspace: calls that need no larger one leave it where it is (captured graphs of earlier calls hold its address),
an error that has not been reported yet outlives its growth, and its first use waits for its clearing whatever stream the
call is on."""
from __future__ import annotations

import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


def on_device(c):
    return [t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias)]


def error(out, c):
    s = c.shape
    ref = torch.from_numpy(oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8))
    return float((out.double().cpu() - ref).abs().max() / ref.abs().max())


# the captured call, then calls of other kernel families whose workspace is smaller; the last has more planes than the arrival
# counters allocated with the workspace are for
CAPTURED = [(2, 8, 64, 64, 128, 3, "f32"), (1, 8, 64, 64, 64, 3, "f32"), (2, 8, 20, 24, 64, 5, "bf16")]
LATER = [(2, 4, 14, 14, 64, 3, "bf16"), (1, 4, 24, 24, 64, 3, "bf16"), (1, 2, 9, 9, 48, 3, "bf16"), (1, 2, 24, 20, 64, 5, "bf16"),
         (1, 2, 9, 9, 32, 5, "f32"), (300, 1, 7, 7, 32, 3, "bf16")]


@pytest.mark.parametrize("captured", CAPTURED, ids=lambda c: "x".join(map(str, c)))
def test_captured_forward_survives_smaller_calls_of_every_family(captured):
    from paper_2211_10526_b200 import CastlingAttn, binding
    first, new = (workloads.custom_call(*captured, seed=1900 + i) for i in range(2))
    s = first.shape
    args = on_device(first)
    out = torch.empty_like(args[0])

    def size(shape):
        B, H, gh, gw, d, _, dtype = shape
        return binding.castling_attn_workspace_bytes(B, H, gh, gw, d, binding.CASTLING_F32 if dtype == "f32" else binding.CASTLING_BF16)
    later = [x for x in LATER if x[5] == s.ksize and size(x) <= size(captured)]
    assert len(later) >= 2
    with CastlingAttn(ksize=s.ksize) as attn:
        attn.forward(*args, s.gridH, s.gridW, out=out)
        torch.cuda.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            attn.forward(*args, s.gridH, s.gridW, out=out)
        for shape in later:
            c = workloads.custom_call(*shape, seed=1910 + sum(shape[:6]))
            got = attn.forward(*on_device(c), c.shape.gridH, c.shape.gridW)
            torch.cuda.synchronize()
            assert error(got, c) <= 2e-2
            for dst, src in zip(args, on_device(new)):
                dst.copy_(src)
            out.zero_()
            graph.replay()
            torch.cuda.synchronize()
            assert error(out, new) <= (1e-5 if captured[6] == "f32" else 2e-2)
        assert attn.device_status() == (0, 0)
        del graph


def test_unreported_status_outlives_the_growth_of_the_workspace():
    from paper_2211_10526_b200 import CastlingAttn, binding
    c = workloads.custom_call(2, 8, 64, 64, 64, 3, "bf16", seed=1920)
    with CastlingAttn() as attn:
        assert binding.castling_attn_selftest_wait(attn.handle, 2000) == binding.OK
        attn.forward(*on_device(c), 64, 64)
        torch.cuda.synchronize()
        assert attn.device_status() == (binding.ERR_DEVICE, 16)
        assert attn.device_status() == (0, 0)
        out = attn.forward(*on_device(c), 64, 64)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    assert error(out, c) <= 2e-2


@pytest.mark.parametrize("shape", [(2, 8, 64, 64, 64, 3, "bf16"), (1, 2, 33, 64, 64, 3, "bf16")], ids=lambda c: "x".join(map(str, c)))
def test_first_call_on_a_stream_of_its_own_while_the_default_stream_is_busy(shape):
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(*shape, seed=1930)
    args = on_device(c)
    busy = torch.randn(4096, 4096, device="cuda:0")
    stream = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(3):
        with CastlingAttn() as attn:
            busy @ busy
            with torch.cuda.stream(stream):
                out = attn.forward(*args, c.shape.gridH, c.shape.gridW)
            torch.cuda.synchronize()
            assert attn.device_status() == (0, 0)
        assert error(out, c) <= 2e-2
