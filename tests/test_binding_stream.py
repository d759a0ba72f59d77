"""The binding's stream handle where torch lacks the private names it prefers."""

import types

import pytest

torch = pytest.importorskip("torch")

from paper_1806_06698_gb300 import syev3  # noqa: E402


@pytest.mark.parametrize("name", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_public_call_without_the_private_names(monkeypatch, name):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=42))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 7, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    assert syev3._stream(None) == 7
    monkeypatch.delattr(torch._C, name)
    assert syev3._stream(None) == 42


def test_a_given_stream_is_taken():
    assert syev3._stream(types.SimpleNamespace(cuda_stream=5)) == 5
