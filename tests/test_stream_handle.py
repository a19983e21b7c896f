"""The stream handle that the binding passes on: the current stream's, with and
without torch's private shortcut to it, or the caller's own."""
from types import SimpleNamespace

import torch

from paper_2609_02897_gb300 import build


def test_stream_handle(monkeypatch):
    build.build()
    from paper_2609_02897_gb300 import asd
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=1234))
    monkeypatch.setattr(asd, "_raw_stream", None)
    assert asd._stream(None) == 1234
    monkeypatch.setattr(asd, "_raw_stream", lambda device: 100 + device)
    assert asd._stream(None) == 103
    assert asd._stream(77) == 77
    assert asd._stream(SimpleNamespace(cuda_stream=55)) == 55
