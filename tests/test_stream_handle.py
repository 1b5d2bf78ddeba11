"""The current stream's handle, with and without torch's private functions for it."""

import types

import pytest
import torch

import paper_2607_28699_gb300 as wc


@pytest.fixture
def current(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))


def test_private_functions_give_the_handle(current, monkeypatch):
    monkeypatch.setattr(wc, "_raw_device", lambda: 3)
    monkeypatch.setattr(wc, "_raw_stream", lambda device: 100 + device)
    assert wc._stream(None) == 103


@pytest.mark.parametrize("missing", ["_raw_stream", "_raw_device"])
def test_a_torch_without_them_gives_the_stream_objects(current, monkeypatch, missing):
    monkeypatch.setattr(wc, "_raw_device", lambda: 3)
    monkeypatch.setattr(wc, "_raw_stream", lambda device: 100 + device)
    monkeypatch.setattr(wc, missing, None)
    assert wc._stream(None) == 1234


def test_before_cuda_is_initialized_and_with_an_explicit_stream(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=55))
    assert wc._stream(None) == 55
    assert wc._stream(types.SimpleNamespace(cuda_stream=77)) == 77
