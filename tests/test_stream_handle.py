"""fdas._stream(None): torch's current stream, with and without torch's raw-handle query."""
import types

import pytest

torch = pytest.importorskip("torch")
from paper_1711_10855_gb300 import fdas


@pytest.mark.parametrize("has_raw", [True, False])
def test_current_stream_handle(monkeypatch, has_raw):
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: types.SimpleNamespace(cuda_stream=4096))
    if has_raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", {3: 4096}.__getitem__, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(fdas, "_raw_stream", None)
    assert fdas._stream(None) == 4096
    assert fdas._stream(None) == 4096   # the kept query
    assert fdas._stream(7) == 7
    assert fdas._stream(types.SimpleNamespace(cuda_stream=11)) == 11
