"""The stream that plan calls run on by default (no GPU)."""
import types

import pytest

torch = pytest.importorskip("torch")


def test_current_stream_without_the_private_call(monkeypatch):
    from paper_2506_04489_gb300 import build
    build.build()
    from paper_2506_04489_gb300.plan import _stream_handle
    current = types.SimpleNamespace(cuda_stream=0x1234)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device=None: current)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert _stream_handle(None) == 0x1234
    assert _stream_handle(types.SimpleNamespace(cuda_stream=7)) == 7
