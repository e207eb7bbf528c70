"""Kernels whose waits can run out are launched only where a status word can tell: a band's apply pass in fp32 takes one on its
first call, and runs the kernels without waits where it cannot have one (during a capture, under a workspace cap)."""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu

SHAPE = (1, 2, 24, 33, 64, 3, "f32")


def kernels(attn, args):
    from paper_2211_10526_b200 import binding
    binding.castling_attn_set_profiling(attn.handle, True)
    out = attn.shard_apply(*args)
    names = [n for n, _ in binding.castling_attn_kernel_times(attn.handle)]
    binding.castling_attn_set_profiling(attn.handle, False)
    return out, names


def test_apply_pass_in_fp32_on_a_fresh_handle():
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(*SHAPE, seed=1950)
    s = c.shape
    q, k, v, w, b = (t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    with CastlingAttn() as attn:
        state = attn.shard_state(k, v)
        want = attn.forward(q, k, v, w, b, s.gridH, s.gridW)
    args = (q, v, w, b, state, s.gridH, s.gridW, 0, 0)
    scale = float(want.abs().max())
    with CastlingAttn() as attn:
        out, names = kernels(attn, args)
        assert names == ["f32_apply"] and float((out - want).abs().max()) <= 1e-5 * scale
        assert attn.device_status() == (0, 0)
    with CastlingAttn(max_workspace=64) as attn:
        out, names = kernels(attn, args)
        assert names == ["simt_apply"] and float((out - want).abs().max()) <= 1e-5 * scale
    with CastlingAttn() as attn:
        out = torch.zeros_like(want)
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph):
            attn.shard_apply(*args, out=out)
        graph.replay()
        torch.cuda.synchronize()
        assert float((out - want).abs().max()) <= 1e-5 * scale
        del graph
