"""Exact angular kernel on the tensor cores where tiles of keys with large cosines follow tiles without: a warp that has met a large one stays
with the general weight function for a while and then looks again.  Planes of up to 40 tiles with large cosines in one of them, in some, in the last,
against the float64 oracle; and each plane alone has to give what it gives among others, bit for bit.

Bound: as where the two forms are tested pair by pair: a cosine of unit rows rounded to bf16 is off by at most 2^-8, a weight and an
output by 2^-9 of themselves, the approximation of arccos by 1e-4.
"""
from __future__ import annotations

import numpy as np
import pytest
import torch

import oracle
import workloads
from test_gpu_weight_branches import cosines

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tiles", [(0,), (3, 17), (5, 30, 39), tuple(range(1, 40, 2))], ids=lambda t: "_".join(map(str, t[:4])))
def test_tiles_with_large_cosines(tiles):
    from paper_2211_10526_b200 import CastlingAttn
    gh, gw = 64, 79   # 39.5 tiles
    c = workloads.custom_call(1, 2, gh, gw, 64, 3, "bf16", seed=91)
    q, k = c.q.float(), c.k.float()
    unit = lambda t: t / t.norm(dim=-1, keepdim=True)
    for t in tiles:   # some keys of these tiles lie near single queries of many tiles
        at = slice(t * 128 + 5, min((t + 1) * 128, gh * gw), 7)
        k[:, 0, at] = 0.9 * unit(q[:, 0, 11::131][:, :k[:, 0, at].shape[1]]) + 0.44 * unit(k[:, 0, at])
    k = k.to(torch.bfloat16)
    dev = torch.device("cuda:0")
    args = [t.to(dev) for t in (c.q, k, c.v, c.dw_weight, c.dw_bias)]
    with CastlingAttn(ksize=3, exact_kernel=True, force_path=2) as attn:
        out = attn.forward(*args, gh, gw)
        alone = [attn.forward(*(t[:, h:h + 1].contiguous() for t in args[:3]), args[3][64 * h:64 * h + 64], args[4][64 * h:64 * h + 64], gh, gw) for h in range(2)]
        torch.cuda.synchronize()
        assert attn.device_status() == (0, 0)
    assert torch.equal(out, torch.cat(alone, dim=1)), "a plane's output depends on the planes beside it"
    got = out.double().cpu().numpy()
    ref = oracle.forward_matrix(c.q, k, c.v, c.dw_weight, c.dw_bias, gh, gw, 3, threads=8, kernel=oracle.KERNEL_EXACT)
    for h in range(2):
        x = cosines(c.q[0, h], k[0, h])
        w = lambda y: 1 - np.arccos(np.clip(y, -1, 1)) / np.pi
        dw = np.maximum(w(x + 2.0 ** -8) - w(x), w(x) - w(x - 2.0 ** -8)) + 2.0 ** -9 * w(x) + 1e-4 / np.pi
        bound = dw @ np.abs(c.v[0, h].double().numpy()) + 2.0 ** -9 * np.abs(ref[0, h]) + 1e-6
        err = np.abs(got[0, h] - ref[0, h])
        assert np.all(err <= bound), f"head {h}: largest error over its bound: {float(np.max(err / bound)):.2f}"
