"""When build() compiles again."""
import torch

from paper_2303_11257_b200 import build as B


def test_a_binding_for_another_torch_is_stale(monkeypatch):
    from paper_2303_11257_b200 import _binding
    B.build()
    assert _binding.built_for == B.built_for() and not B._stale()
    monkeypatch.setattr(torch, "__version__", "2.1")
    assert B._stale()
    monkeypatch.undo()
    monkeypatch.setattr(B.sys, "version_info", (3, 9))
    assert B._stale()
