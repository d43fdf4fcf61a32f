"""The handle of the current stream, with and without torch's private call for it."""
import types

import pytest

torch = pytest.importorskip("torch")


def test_without_the_private_call(monkeypatch):
    import paper_1511_05690_gb300 as pn
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda: types.SimpleNamespace(cuda_stream=0x1234))
    assert pn._stream_ptr(None).value == 0x1234


def test_with_the_private_call(monkeypatch):
    import paper_1511_05690_gb300 as pn
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 0x100 + dev,
                        raising=False)
    assert pn._stream_ptr(None).value == 0x103


def test_a_stream_of_the_caller():
    import paper_1511_05690_gb300 as pn
    assert pn._stream_ptr(types.SimpleNamespace(cuda_stream=7)).value == 7
