"""The calls of a step read the current stream's handle through functions of torch that are not public; without them they take the
public way."""
import types

import torch

import paper_2607_18002_b200 as moe


def _fake_torch(monkeypatch, **functions):
    monkeypatch.setattr(torch.cuda, "init", lambda: None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=11))
    for name in ("_cuda_getDevice", "_cuda_getCurrentRawStream"):
        monkeypatch.delattr(torch._C, name, raising=False)
        if name in functions:
            monkeypatch.setattr(torch._C, name, functions[name], raising=False)
    monkeypatch.setattr(moe, "_read_stream", None)


def test_public_way_without_the_private_functions(monkeypatch):
    _fake_torch(monkeypatch)
    assert moe.Context._stream(None) == 11
    _fake_torch(monkeypatch, _cuda_getDevice=lambda: 3)
    assert moe.Context._stream(None) == 11
    assert moe.Context._stream(types.SimpleNamespace(cuda_stream=5)) == 5


def test_private_functions_are_asked_each_time(monkeypatch):
    device = [2]
    _fake_torch(monkeypatch, _cuda_getDevice=lambda: device[0], _cuda_getCurrentRawStream=lambda d: 100 + d)
    assert moe.Context._stream(None) == 102
    device[0] = 4
    assert moe.Context._stream(None) == 104
