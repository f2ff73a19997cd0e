"""The module that marshals a step's arguments belongs to one Python and one torch: with another torch it is neither fresh nor loaded."""
import pytest
import torch

from paper_2507_07114_b200 import binding, build


def test_another_torch_wants_another_module(monkeypatch):
    build.build()
    path = build.marshal_path()
    assert not build._stale(path)
    monkeypatch.setattr(torch, "__version__", "2.0.0+elsewhere")
    other = build.marshal_path()
    assert other != path and build._stale(other)
    monkeypatch.setattr(binding, "_native", None)
    monkeypatch.setattr(binding, "_lib", None)
    with pytest.raises(FileNotFoundError, match="2.0.0"):
        binding.load_library()
