"""Tensors without storage (inside vmap, fake ones) are refused with an exception, and the handle serves the next call."""
from __future__ import annotations

import pytest
import torch

import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2, 3, 6, 8, 64, 3, "bf16"), (2, 3, 6, 8, 32, 3, "f32")], ids=lambda c: "x".join(map(str, c)))
def test_refused_with_an_exception(shape):
    from paper_2211_10526_b200 import CastlingAttn
    from torch._subclasses.fake_tensor import FakeTensorMode
    c = workloads.custom_call(*shape, seed=2100)
    q, k, v, w, b = (t.to("cuda:0") for t in (c.q, c.k, c.v, c.dw_weight, c.dw_bias))
    with CastlingAttn() as attn:
        want = attn.forward(q, k, v, w, b, 6, 8)
        with pytest.raises(Exception):
            torch.func.vmap(lambda x: attn.forward(x, k, v, w, b, 6, 8))(torch.stack([q, q]))
        with pytest.raises(Exception):
            torch.func.vmap(lambda x: attn.forward(q, k, v, w, x, 6, 8))(torch.stack([b, b]))
        with FakeTensorMode() as mode:
            fake = [mode.from_tensor(t) for t in (q, k, v, w, b)]
            with pytest.raises(Exception):
                attn.forward(*fake, 6, 8)
        assert torch.equal(attn.forward(q, k, v, w, b, 6, 8), want)
