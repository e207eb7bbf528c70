"""Width-32 grids that fit no 128-byte rows, pinned to the tensor-core kernels: taken whatever the number of planes, down to one
token, against the float64 oracle (2e-2 of the largest output, as for every bf16 shape)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads

pytestmark = pytest.mark.gpu

CASES = [(1, 1, 1, 1, 32, 3), (1, 1, 7, 7, 32, 3), (2, 2, 7, 7, 32, 5), (1, 3, 1, 31, 32, 3), (1, 1, 23, 25, 32, 3), (1, 2, 33, 21, 32, 5),
         (1, 1, 9, 1, 32, 5), (1, 1, 3, 301, 32, 3)]


@pytest.mark.parametrize("rownorm", [False, True], ids=["core", "rownorm"])
@pytest.mark.parametrize("shape", CASES, ids=lambda c: "x".join(map(str, c)))
def test_any_number_of_planes(shape, rownorm):
    from paper_2211_10526_b200 import CastlingAttn, binding
    c = workloads.custom_call(*shape, "bf16", seed=2150 + sum(shape))
    s = c.shape
    args = [t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias)]
    with CastlingAttn(ksize=s.ksize, force_path=binding.PATH_TENSOR, normalize_rows=rownorm) as attn:
        out = attn.forward(*args, s.gridH, s.gridW)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0) and attn.last_path()[0] == binding.PATH_TENSOR
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, s.gridH, s.gridW, s.ksize, threads=8)
    err = float(np.max(np.abs(out.double().cpu().numpy() - ref)) / np.max(np.abs(ref)))
    assert err <= 2e-2, f"max-rel error {err:.3e}"
