"""A floor whose square is below the smallest float, on every kernel family: tiles are filled up with rows of zeros, which stay
zeros, and so does a zero row of the input (cosine 0 with everything)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

CASES = [(2, 3, 7, 9, 32, 3, "f32"), (2, 3, 33, 31, 64, 5, "f32"), (1, 2, 9, 9, 48, 3, "f32"), (40, 4, 5, 5, 32, 3, "f32"),
         (60, 8, 7, 7, 32, 3, "bf16"), (8, 8, 25, 39, 32, 5, "bf16"), (4, 12, 14, 14, 64, 3, "bf16"), (2, 2, 24, 21, 64, 3, "bf16"),
         (2, 3, 5, 7, 48, 3, "bf16"), (2, 4, 24, 20, 32, 3, "bf16")]


@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_zero_rows_stay_zero(case, rownorm):
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(*case, seed=2000 + sum(case[:6]))
    s = c.shape
    c.q[0, 0, 3] = 0
    c.k[-1, -1, 5] = 0
    args = [t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias)]
    with CastlingAttn(ksize=s.ksize, eps=1e-30, normalize_rows=rownorm) as attn:
        out = attn.forward(*args, s.gridH, s.gridW)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8)
    got = out.double().cpu().numpy()
    assert np.all(np.isfinite(got))
    assert float(np.max(np.abs(got - ref)) / np.max(np.abs(ref))) <= (1e-5 if s.dtype == "f32" else 2e-2)


@pytest.mark.parametrize("variant", [{"exact_kernel": True}, {"sparse_eps": 0.01}], ids=["exact", "masked"])
def test_explicit_weights(variant):
    from paper_2211_10526_b200 import CastlingAttn
    c = workloads.custom_call(2, 3, 9, 21, 64, 3, "bf16", seed=2050)
    args = [t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias)]
    with CastlingAttn(**variant) as attn:
        want = attn.forward(*args, 9, 21)
    with CastlingAttn(eps=1e-30, **variant) as attn:
        assert torch.equal(attn.forward(*args, 9, 21), want)
