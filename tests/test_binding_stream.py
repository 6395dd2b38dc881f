"""The stream handle that a call passes on, with and without torch's undocumented
accessor of the raw handle (a stand-in for torch: no GPU)."""
from types import SimpleNamespace as NS

from paper_2412_02413_gb300 import pam


def _torch(**private):
    return NS(_C=NS(**private), cuda=NS(current_device=lambda: 1, current_stream=lambda: NS(cuda_stream=42)))


def test_stream_handle(monkeypatch):
    monkeypatch.setattr(pam, "_torch", _torch(_cuda_getCurrentRawStream=lambda device: 100 + device))
    assert pam._stream_ptr() == 101
    monkeypatch.setattr(pam, "_torch", _torch())
    assert pam._stream_ptr() == 42
    assert pam._stream_ptr(NS(cuda_stream=7)) == 7
