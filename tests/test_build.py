"""When the library and its extensions are rebuilt, and what a failed build leaves behind (no GPU needed)."""
import torch

from paper_2608_15522_b200 import build


def test_extension_of_another_pytorch_is_rebuilt(monkeypatch):
    """The allocating extension is bound to the PyTorch that it was compiled against, which file times do not tell."""
    build.build_library()
    assert not build._stale()
    monkeypatch.setattr(torch, "__version__", "0.0.1")
    assert build._stale()
