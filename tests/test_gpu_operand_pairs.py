"""Width-32 bf16 calls that the tensor-core kernels take with operand pairs (unit keys and scaled states as two bf16: grids that
the packed rows do not fit, and planes under 96 tokens) are as precise as fp32 arithmetic: what is left is the rounding of the
output to bf16.  Bound: a pair leaves 2^-17 of an operand, which adds (2^-17 / 2^-9)^2 < 2e-5 to that rounding's relative error
(2-norm); 2e-3 covers that and the elements that fall on the other side of a rounding boundary.  Operands of a single bf16
miss it (1.2e-2 above)."""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_narrow_rows import views

pytestmark = pytest.mark.gpu

#        B, H, gridH, gridW, ksize, layout, prefix, row sums
CASES = [(64, 8, 7, 7, 3, "heads", 0, False), (40, 6, 8, 8, 5, "heads", 0, False), (8, 3, 16, 16, 3, "tokens", 0, False),
         (4, 5, 1, 257, 3, "heads", 0, False), (5, 3, 16, 31, 5, "heads", 3, False), (9, 9, 15, 17, 3, "heads", 1, False),
         (8, 8, 25, 38, 5, "heads", 1, False), (2, 3, 121, 131, 3, "heads", 0, False), (5, 3, 17, 31, 5, "tokens", 2, False),
         (64, 8, 7, 7, 3, "heads", 0, True), (40, 6, 8, 8, 5, "heads", 0, True), (9, 9, 9, 9, 5, "fused", 2, True)]


@pytest.mark.parametrize("case", CASES, ids=lambda c: "x".join(map(str, c)))
def test_error_is_the_rounding_of_the_output(case):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, gh, gw, ks, layout, prefix, rownorm = case
    c = workloads.custom_call(B, H, 1, prefix + gh * gw, 32, ks, "bf16", seed=1800 + gh + gw + ks, qk_lognormal_sigma=0.5)
    dev = torch.device("cuda:0")
    q, k, v, out = views(c, layout, dev)
    with CastlingAttn(ksize=ks, prefix_tokens=prefix, normalize_rows=rownorm) as attn:
        attn.forward(q, k, v, c.dw_weight.to(dev), c.dw_bias.to(dev), gh, gw, out=out)
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
        assert attn.last_path()[0] == 2
    ref = (oracle.forward_rownorm if rownorm else oracle.forward)(c.q, c.k, c.v, c.dw_weight, c.dw_bias, gh, gw, ks, threads=8,
                                                                  prefix=prefix)
    ref = torch.from_numpy(np.asarray(ref, dtype=np.float64))
    rounding = float((ref.to(torch.bfloat16).double() - ref).norm())
    err = float((out.double().cpu() - ref).norm())
    assert err <= (1 + 2e-3) * rounding, f"{err / rounding:.5f} of the rounding of the output"
