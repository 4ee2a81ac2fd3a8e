"""The binding's default stream: torch's public call wherever the private one it prefers is missing."""
import types

import pytest

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("missing", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_private_functions(monkeypatch, missing):
    from paper_1810_06250_gb300 import _binding
    monkeypatch.delattr(torch._C, missing, raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    assert _binding._stream(None) == 1234
    assert _binding._stream(77) == 77
