"""Which exception forward_host raises for what (its checks need no device)."""
from __future__ import annotations

import pytest
import torch


def _call(**change):
    from paper_2211_10526_b200 import CastlingAttn
    attn = CastlingAttn.__new__(CastlingAttn)   # no handle: the checks come before the library is called
    attn.ksize, attn.prefix_tokens = 3, 0
    t = {n: torch.zeros(1, 2, 12, 32) for n in ("q", "k", "v", "out")}
    t.update(w=torch.zeros(64, 3, 3), bias=torch.zeros(64))
    t.update(change)
    return attn._check_host(t["q"], t["k"], t["v"], t["w"], t["bias"], t["out"], 3, 4)


@pytest.mark.parametrize("change,error", [
    ({"bias": torch.zeros(64, dtype=torch.bfloat16)}, ValueError),
    ({"bias": torch.zeros(128)[::2]}, ValueError),
    ({"bias": torch.zeros(32)}, ValueError),
    ({"bias": torch.zeros(64, dtype=torch.bfloat16), "k": torch.zeros(1, 2, 12, 32, dtype=torch.bfloat16)}, ValueError),
    ({"k": torch.zeros(1, 2, 12, 32, dtype=torch.bfloat16)}, TypeError),
    ({"w": torch.zeros(64, 3, 3, dtype=torch.float64)}, TypeError),
    ({"k": torch.zeros(1, 2, 12, 32, dtype=torch.bfloat16), "w": torch.zeros(64, 3, 3).transpose(1, 2)}, ValueError),
    ({"v": torch.zeros(1, 2, 32, 12).transpose(2, 3)}, ValueError),
    ({"out": torch.zeros(1, 2, 12, 32, device="meta")}, ValueError),
    ({"q": torch.zeros(1, 2, 12, 16)}, ValueError)])
def test_exception(change, error):
    with pytest.raises(error):
        _call(**change)


def test_accepted():
    assert _call() == (1, 2, 12, 32) and _call(bias=None) == (1, 2, 12, 32)
