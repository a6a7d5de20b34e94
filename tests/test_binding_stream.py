"""The stream handle that the calls are enqueued on, with a torch that has the private shortcuts and with one that lacks them."""
import types

import pytest
import torch

from paper_2412_16187_b200 import binding


def test_an_explicit_stream_is_taken_as_it_is():
    assert binding._stream(types.SimpleNamespace(cuda_stream=77)) == 77


@pytest.mark.parametrize("gone", ["_cuda_getCurrentRawStream", "_cuda_getDevice"])
def test_current_stream_without_the_private_functions(monkeypatch, gone):
    monkeypatch.setattr(torch._C, "_cuda_getDevice", lambda: 0, raising=False)
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 4711 + device, raising=False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=42))
    assert binding._stream() == 4711
    monkeypatch.delattr(torch._C, gone)
    assert binding._stream() == 42
