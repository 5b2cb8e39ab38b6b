"""The binding's stream handle does not depend on PyTorch's private names."""
import types

import pytest

torch = pytest.importorskip("torch")

from paper_2406_06385_gb300 import lrqat as LQ


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_public_stream_without_the_private_names(missing, monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    for name in ("_cuda_getCurrentRawStream", "_cuda_getDevice"):
        monkeypatch.setattr(torch._C, name, lambda *a: 5, raising=False)
    assert LQ._stream(None) == 5
    monkeypatch.delattr(torch._C, missing)
    assert LQ._stream(None) == 77
