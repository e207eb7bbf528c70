"""fp32 planes of one or two columns, of one long row and of a few tokens: the kernels that each call takes (those that were measured as the faster ones), and
its output against the float64 oracle.  Bound: sums of at most 256 fp32 terms, 1e-5 of the largest output, as for all short fp32 planes.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_narrow_rows import views

pytestmark = pytest.mark.gpu

TWO, ONE, CORES = ["f32_state", "f32_apply"], ["f32_plane"], ["simt_fused"]
#        B, H, gridH, gridW, d, ksize, layout, prefix, kernels (None: not told apart by their names)
CASES = [(5, 4, 64, 1, 64, 3, "heads", 0, TWO), (5, 4, 64, 1, 32, 5, "tokens", 1, TWO), (37, 4, 128, 1, 32, 3, "heads", 0, TWO), (12, 4, 251, 1, 32, 3, "fused", 2, TWO),
         (50, 3, 64, 1, 32, 3, "heads", 0, CORES), (50, 3, 64, 1, 64, 3, "heads", 0, CORES), (90, 1, 254, 1, 32, 3, "heads", 1, TWO), (100, 1, 254, 1, 32, 3, "heads", 1, None), (100, 1, 256, 1, 32, 3, "heads", 0, None),
         (5, 4, 30, 2, 64, 3, "heads", 0, TWO), (16, 4, 30, 2, 64, 5, "tokens", 0, ONE), (100, 4, 25, 2, 32, 3, "heads", 0, CORES), (75, 4, 60, 2, 32, 3, "heads", 1, ONE),
         (75, 4, 25, 2, 64, 3, "heads", 0, CORES), (32, 3, 4, 4, 32, 3, "heads", 0, CORES), (32, 3, 3, 6, 32, 3, "heads", 0, ONE), (2, 4, 1, 250, 32, 3, "heads", 0, None),
         (2, 4, 1, 128, 64, 3, "tokens", 0, None), (2, 4, 2, 128, 64, 3, "heads", 0, None), (2, 4, 1, 192, 32, 5, "heads", 0, None), (2, 4, 1, 193, 32, 5, "heads", 0, None)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c[:8])))
def test_thin_planes(case):
    from paper_2211_10526_b200 import CastlingAttn, binding
    B, H, gh, gw, d, ks, layout, prefix, kernels = case
    dev = torch.device("cuda:0")
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, d, ks, "f32", seed=2700 + gh + gw, qk_lognormal_sigma=0.5)
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=ks, prefix_tokens=prefix) as attn:
        binding.castling_attn_set_profiling(attn.handle, True)
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        taken = [name for name, _ in binding.castling_attn_kernel_times(attn.handle)]
    assert kernels is None or taken == kernels
    ref = oracle.forward(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8, prefix=prefix)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got)), "an output element was never written"
    err = float(np.max(np.abs(got - ref)) / np.max(np.abs(ref)))
    assert err <= 1e-5, f"max-rel error {err:.3e}"
