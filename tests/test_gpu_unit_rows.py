"""Unit rows of K, bit for bit: a key element is its value times 1 / ||k||, that factor in fp32, with one rounding to bf16.

Keys hold small integers, so that a row's sum of squares is exact in any order.  The factor and the product are then off by at most 2^-23 and
2^-24, so an element is the rounding of x / ||k||, or that of a number within 2^-22 of it.  Values are unit vectors, which single out one key each: the state holds the unit rows themselves, and a
query that is a unit vector brings a row of the scaled state out.
"""
from __future__ import annotations

import math

import pytest
import torch

pytestmark = pytest.mark.gpu


def keys(B, H, N, d, live, seed):
    """Integer rows, zero from token `live` on, and the lowest and the highest unit rows that one rounding allows."""
    gen = torch.Generator().manual_seed(seed)
    k = torch.randint(-127, 128, (B, H, N, d), generator=gen).double()
    k[:, :, live:] = 0
    unit = k / k.norm(dim=-1, keepdim=True).clamp_min(1e-12)
    return k.to(torch.bfloat16), [(unit * (1 + s * 2.0 ** -22)).to(torch.bfloat16) for s in (-1, 1)]


@pytest.mark.parametrize("N", [64, 200, 1500])
def test_state_holds_the_unit_rows(N):
    from paper_2211_10526_b200 import CastlingAttn
    B, H, d = 4, 8, 64
    k, unit = keys(B, H, N, d, N, 41 + N)
    v = torch.zeros(B, H, N, d, dtype=torch.bfloat16)
    v[:, :, torch.arange(d), torch.arange(d)] = 1
    with CastlingAttn() as attn:
        state = attn.shard_state(k.cuda(), v.cuda())
        assert attn.device_status() == (0, 0)
        assert attn.last_path()[0] == 2
    got = state[:, :d * d].reshape(B, H, d, d).cpu()
    low, high = (u[:, :, :d].float().transpose(-1, -2) for u in unit)
    assert torch.all((got == low) | (got == high)), f"{int(((got != low) & (got != high)).sum())} elements rounded another way"


#        gridH, gridW, d: one kernel per plane (both CTA shapes), and state and apply kernels
@pytest.mark.parametrize("grid", [(8, 16, 64), (14, 14, 64), (8, 16, 32), (14, 14, 32), (24, 24, 32), (24, 32, 64)], ids=lambda g: "x".join(map(str, g)))
def test_output_holds_the_unit_rows(grid):
    from paper_2211_10526_b200 import CastlingAttn
    gh, gw, d = grid
    B, H, N = 8, 4, gh * gw
    k, unit = keys(B, H, N, d, d, 43 + N)
    eye = torch.eye(d)
    v = torch.zeros(B, H, N, d)
    v[:, :, :d], v[:, :, d:2 * d] = eye, -eye   # the second block, on keys of zeros, takes the token sum away
    q = eye.repeat(N // d + 1, 1)[:N].expand(B, H, N, d)
    with CastlingAttn(force_path=2) as attn:
        out = attn.forward(q.to(torch.bfloat16).contiguous().cuda(), k.cuda(), v.to(torch.bfloat16).cuda(),
                           torch.zeros(H * d, 3, 3, dtype=torch.bfloat16, device="cuda"), None, gh, gw)
        assert attn.device_status() == (0, 0)
    # S', rows by key feature
    low, high = ((u[:, :, :d].float().transpose(-1, -2) * (1 / math.pi)).to(torch.bfloat16).repeat(1, 1, N // d + 1, 1)[:, :, :N] for u in unit)
    got = out.cpu()
    assert torch.all((got == low) | (got == high)), f"{int(((got != low) & (got != high)).sum())} elements rounded another way"
