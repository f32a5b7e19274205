"""The binding's stream handle: the given stream's, else the current stream's, with
torch's private call for it and without (a torch may drop it).  No device."""
import types

import pytest

from paper_2503_13756_gb300 import swalign

torch = pytest.importorskip("torch")


def test_given_stream():
    assert swalign._stream(types.SimpleNamespace(cuda_stream=5)) == 5


def test_current_stream_with_and_without_the_private_call(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 40 + d, raising=False)
    assert swalign._stream() == 43
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert swalign._stream() == 77
