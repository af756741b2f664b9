"""The stream handle of the device calls: PyTorch's internal call where it has it, else the
public one (PyTorch's internal names may go)."""
import types

import pytest


@pytest.mark.parametrize("internal", [True, False])
def test_stream_handle(monkeypatch, internal):
    import torch
    from paper_1801_10277_gb300 import celeste
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 1)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=0x51))
    if internal:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 0x50 + d, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert celeste.Problem._stream().value == 0x51
