"""The handle of the stream a call runs on: the caller's, or torch's current one, with or without torch's
private way to ask for it (CPU, a stand-in for torch)."""
from types import SimpleNamespace

import pytest

import paper_2508_06710_gb300 as rb


@pytest.mark.parametrize("private", [True, False])
def test_stream_handle(monkeypatch, private):
    fake = SimpleNamespace(_C=SimpleNamespace(), cuda=SimpleNamespace(
        current_device=lambda: 3, current_stream=lambda: SimpleNamespace(cuda_stream=0x5000)))
    if private:
        fake._C._cuda_getCurrentRawStream = lambda device: 0x4000 + device
    monkeypatch.setattr(rb, "_torch", lambda: fake)
    assert rb._stream() == (0x4003 if private else 0x5000)
    assert rb._stream(SimpleNamespace(cuda_stream=0x77)) == 0x77
