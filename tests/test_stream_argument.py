"""The stream that a call is queued on: the given one, else torch's current
one, also where torch lacks the call that is only an implementation of its."""
from types import SimpleNamespace

import pytest

torch = pytest.importorskip("torch")

from paper_2003_10558_gb300 import vsr  # noqa: E402


def test_given_stream():
    assert vsr._stream_ptr(SimpleNamespace(cuda_stream=7)) == 7


@pytest.mark.parametrize("private", [True, False])
def test_current_stream(monkeypatch, private):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 2, raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=40))
    if private:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 38 + d, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert vsr._stream_ptr(None) == 40
