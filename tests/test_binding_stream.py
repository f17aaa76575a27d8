"""CPU check of the binding's stream lookup on a torch without the private functions it
prefers (torch._C._cuda_getCurrentRawStream, _cuda_getDevice)."""
import importlib.util
import types

import pytest
import torch

from paper_1609_05344_gb300 import api


@pytest.mark.parametrize("private", [True, False])
def test_stream_handle_with_and_without_private_functions(monkeypatch, private):
    for name, value in (("_cuda_getCurrentRawStream", lambda device: 70 + device), ("_cuda_getDevice", lambda: 3)):
        monkeypatch.setattr(torch._C, name, value, raising=False)
        if not private:
            monkeypatch.delattr(torch._C, name)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 5)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=99))
    spec = importlib.util.spec_from_file_location("paper_1609_05344_gb300.api_copy", api.__file__)
    copy = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(copy)
    assert copy._stream() == (73 if private else 99)
    assert copy._stream(types.SimpleNamespace(cuda_stream=42)) == 42
    with pytest.raises(ValueError):
        copy._require_cuda(torch.zeros(1), "t")
