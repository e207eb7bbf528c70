"""The torch-facing module is rebuilt for another torch version, whose C++ interface may differ."""
from __future__ import annotations

import torch


def test_another_torch_version_makes_the_module_stale(monkeypatch):
    from paper_2211_10526_b200 import _torch_call, build
    build.build()
    assert not build._call_stale()
    assert _torch_call.built_against == f"built against torch {torch.__version__}"
    monkeypatch.setattr(torch, "__version__", torch.__version__ + ".post1")
    assert build._call_stale()
    monkeypatch.setattr(torch, "__version__", torch.__version__[:-7])
    assert build._call_stale()
