"""The caller's stream as the binding looks it up (no GPU needed): by torch's raw-stream functions, else by the public Stream
object: where a function is missing and where CUDA is not up (torch then initializes it, or refuses as it always did, for one
in a forked child)."""
from types import SimpleNamespace

import pytest
import torch

import paper_2401_07805_gb300 as evap


@pytest.fixture
def public(monkeypatch):
    calls = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: calls.append(1) or SimpleNamespace(cuda_stream=11))
    return calls


def test_raw_stream(monkeypatch, public):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(evap, "_current_device", lambda: 3)
    monkeypatch.setattr(evap, "_raw_stream", lambda device: 100 + device)
    assert evap._stream() == 103 and not public


@pytest.mark.parametrize("name", ["_raw_stream", "_current_device"])
def test_a_missing_function(monkeypatch, public, name):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(evap, name, None)
    assert evap._stream() == 11 and public == [1]


def test_cuda_not_up(monkeypatch, public):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: False)
    assert evap._stream() == 11 and public == [1]
