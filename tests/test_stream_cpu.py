"""The training wrappers' stream handle (CPU, torch.cuda faked): torch's raw
handle where the release has it, else the public stream object's."""
import types

import pytest

from paper_2409_10729_gb300 import mfc


@pytest.mark.parametrize("raw", [True, False])
def test_stream_of_the_current_device(monkeypatch, raw):
    torch = pytest.importorskip("torch")
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d=None: types.SimpleNamespace(cuda_stream=4000 + d))
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 5000 + d, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert mfc._stream() == (5003 if raw else 4003)
