"""How the binding finds the current stream, without a GPU."""
import types

import pytest
import torch

from paper_2405_01420_gb300 import nb

FAST = ("_cuda_getCurrentRawStream", "_cuda_getDevice")


@pytest.fixture
def initialized(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=77))
    monkeypatch.setattr(torch._C, FAST[0], lambda device: 1000 + device, raising=False)
    monkeypatch.setattr(torch._C, FAST[1], lambda: 3, raising=False)


def test_current_stream_of_the_current_device(initialized):
    assert nb._stream(None) == 1003


@pytest.mark.parametrize("name", FAST)
def test_a_torch_without_the_private_functions(initialized, monkeypatch, name):
    monkeypatch.delattr(torch._C, name)
    assert nb._stream(None) == 77


def test_before_cuda_is_initialized(initialized, monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    assert nb._stream(None) == 77


def test_a_raw_handle_is_passed_on():
    assert nb._stream(5) == 5
