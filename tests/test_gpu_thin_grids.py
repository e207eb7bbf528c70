"""Thin grids (a row, a column, a few rows or columns) on the kernels that walk through a grid in patches, against the float64
oracle, with filters thirty times as large as elsewhere so that the convolution is what is seen.  Bound: 2e-2 of the largest
output for bf16 (operands and output rounded to 2^-9), 1e-5 for fp32."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu


def thin(shape, seed):
    c = workloads.custom_call(*shape, seed=seed)
    c.dw_weight = (c.dw_weight.float() * 30).to(c.dw_weight.dtype)
    c.dw_bias = (c.dw_bias.float() * 20).to(c.dw_bias.dtype)
    return c


def run(c, path, **config):
    from paper_2211_10526_b200 import CastlingAttn
    s = c.shape
    args = [t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias)]
    out = torch.full_like(args[0], float("nan"))
    with CastlingAttn(ksize=s.ksize, **config) as attn:
        attn.forward(*args, s.gridH, s.gridW, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path()[0] == path
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    return got


def worst(got, ref):
    return float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))


@pytest.mark.parametrize("shape", [(1, 2, 1, 600, 64, 3), (1, 2, 600, 1, 64, 3), (1, 2, 2, 331, 64, 5), (1, 2, 3, 700, 64, 3), (2, 2, 1, 40, 64, 5),
                                   (2, 2, 40, 1, 64, 5), (1, 1, 2, 129, 64, 3), (1, 1, 1, 2000, 64, 5), (1, 2, 2000, 1, 64, 5), (1, 2, 7, 90, 64, 3),
                                   (1, 2, 257, 2, 64, 3), (40, 8, 196, 1, 64, 3), (1, 2, 5, 257, 64, 5), (1, 3, 3, 256, 64, 3), (1, 70, 3, 300, 64, 3)],
                         ids=lambda c: "x".join(map(str, c)))
def test_explicit_weights(shape):
    c = thin((*shape, "bf16"), 2200 + sum(shape))
    s = c.shape
    ref = oracle.forward_matrix(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8, kernel=oracle.KERNEL_EXACT)
    assert worst(run(c, 2, exact_kernel=True), ref) <= 2e-2


@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("shape", [(8, 8, 1, 601, 32, 5), (8, 8, 601, 1, 32, 5), (8, 8, 600, 1, 32, 3), (5, 9, 1031, 1, 32, 3), (8, 8, 301, 2, 32, 3)],
                         ids=lambda c: "x".join(map(str, c)))
def test_width_32(shape, rownorm):
    c = thin((*shape, "bf16"), 2300 + sum(shape))
    s = c.shape
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8)
    assert worst(run(c, 2, normalize_rows=rownorm), ref) <= 2e-2


# on both sides of the rule: patches four times (3.5 times) as large as the grid, more of them than run at a time
@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("shape", [(1, 4, 1, 2000, 64, 3), (1, 4, 2000, 1, 64, 5), (4, 12, 2, 331, 64, 3), (4, 12, 331, 4, 64, 3), (4, 12, 331, 5, 64, 5),
                                   (1, 4, 1, 3000, 32, 3), (1, 4, 3000, 1, 32, 5), (4, 12, 641, 7, 32, 3), (4, 12, 641, 8, 32, 3), (4, 12, 1, 501, 128, 3),
                                   (4, 12, 200, 2, 128, 5), (4, 12, 3, 201, 128, 3), (1, 2, 1, 70, 64, 3)],
                         ids=lambda c: "x".join(map(str, c)))
def test_fp32(shape, rownorm):
    c = thin((*shape, "f32"), 2400 + sum(shape))
    s = c.shape
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8)
    assert worst(run(c, 1, normalize_rows=rownorm), ref) <= 1e-5


def test_bands_of_a_thin_grid_in_fp32():
    from paper_2211_10526_b200 import CastlingAttn
    c = thin((4, 12, 400, 1, 64, 3, "f32"), 2500)
    q, k, v, w, b = (t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    out = torch.full_like(q, float("nan"))
    with CastlingAttn() as attn:
        state = attn.shard_state(k, v)
        for y0, y1 in ((0, 150), (150, 400)):
            top, bottom = int(y0 > 0), int(y1 < 400)
            out[:, :, y0:y1] = attn.shard_apply(q[:, :, y0:y1].contiguous(), v[:, :, y0 - top:y1 + bottom].contiguous(), w, b, state,
                                                y1 - y0, 1, top, bottom)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, 400, 1, 3, threads=8)
    assert worst(out.double().cpu().numpy(), ref) <= 1e-5
