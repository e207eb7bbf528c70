"""Masked branch on the tensor cores: the weights of pairs whose probability the mask takes away, bit for bit.  Queries are unit vectors, so
that a cosine is an element of a unit key row, which the contraction keeps whole; values are unit vectors, so that an output is one weight
1/2 + x / pi, rounded to bf16.  Keys hold small integers: their unit rows are off by one rounding and 2^-22 (the factor and the
product in fp32), the weight by its own rounding and 2^-22.
"""
from __future__ import annotations

import math

import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("grid", [(8, 8), (9, 14), (14, 14), (20, 30)], ids=lambda g: f"{g[0]}x{g[1]}")
def test_weight_is_a_half_and_the_cosine_over_pi(grid):
    from paper_2211_10526_b200 import CastlingAttn
    gh, gw = grid
    B, H, d, N = 2, 4, 64, gh * gw
    gen = torch.Generator().manual_seed(61 + N)
    k = torch.randint(-127, 128, (B, H, N, d), generator=gen) * (torch.rand(B, H, N, d, generator=gen) < 0.06)   # a few large cosines a row
    k = k.double()
    q = torch.eye(d).repeat(N // d + 1, 1)[:N].expand(B, H, N, d)
    v = torch.zeros(B, H, N, d)
    v[:, :, :d] = torch.eye(d)
    with CastlingAttn(sparse_eps=1.0, force_path=2) as attn:
        out = attn.forward(*(t.to(torch.bfloat16).contiguous().cuda() for t in (q, k, v)),
                           torch.zeros(H * d, 3, 3, dtype=torch.bfloat16, device="cuda"), None, gh, gw)
        assert attn.device_status() == (0, 0)
    got = out.cpu()
    unit = k / k.norm(dim=-1, keepdim=True).clamp_min(1e-12)
    right = torch.zeros(got.shape, dtype=torch.bool)
    for a in (-1, 1):
        x = (unit * (1 + a * 2.0 ** -22)).to(torch.bfloat16).double()[:, :, :d].transpose(-1, -2)
        for b in (-1, 1):
            w = ((0.5 + x / math.pi) * (1 + b * 2.0 ** -22)).to(torch.bfloat16)
            right |= got == w.repeat(1, 1, N // d + 1, 1)[:, :, :N]
    assert torch.all(right), f"{int((~right).sum())} weights of {right.numel()} differ"
