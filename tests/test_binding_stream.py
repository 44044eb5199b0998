"""The binding's stream handle: the stream it is given, or the device's current one, with or without
torch's private shortcut to its handle."""
import types

import pytest
import torch

from paper_2606_18954_gb300 import binding


@pytest.mark.parametrize("shortcut", [True, False])
@pytest.mark.parametrize("index", [None, 3])
def test_current_stream(monkeypatch, shortcut, index):
    dev = torch.device("cuda") if index is None else torch.device("cuda", index)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 5)
    monkeypatch.setattr(torch.cuda, "current_stream",
                        lambda d: types.SimpleNamespace(cuda_stream=100 + (5 if d.index is None else d.index)))
    if shortcut:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda i: 100 + i, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert binding._raw_stream(None, dev).value == 100 + (5 if index is None else index)
    assert binding._raw_stream(types.SimpleNamespace(cuda_stream=77), dev).value == 77
