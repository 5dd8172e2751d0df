"""The stream a call without one is queued on: torch's current stream, also
where torch lacks the raw handle's accessors (never the default stream
instead)."""
import types

import pytest

torch = pytest.importorskip("torch")
from paper_2307_12988_gb300 import _binding


def test_current_stream_without_raw_accessors(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert _binding._stream(None) == 77
    assert _binding._stream(5) == 5
    assert _binding._stream(types.SimpleNamespace(cuda_stream=6)) == 6
