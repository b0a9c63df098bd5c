"""The stream handle that a call passes on: the given stream's, torch's current one, and the current one where torch does
not have the private entry that gives it without a Stream object."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2607_14513_gb300 import gsc


def test_given_stream():
    assert gsc._stream(SimpleNamespace(cuda_stream=0x77)).value == 0x77


def test_current_stream(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 0x100 + device, raising=False)
    assert gsc._stream(None).value == 0x103


def test_current_stream_without_the_private_entry(monkeypatch):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=0x55))
    assert gsc._stream(None).value == 0x55
