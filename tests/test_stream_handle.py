"""The stream of a call without one is the current device's current stream, with or without torch's raw accessor."""
import types

import pytest
import torch

from paper_1407_0904_gb300 import binding as B


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream(monkeypatch, raw):
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda dev=None: types.SimpleNamespace(cuda_stream=40 + dev))
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda dev: 40 + dev, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert B._stream_handle(None).value == 43
    assert B._stream_handle(types.SimpleNamespace(cuda_stream=7)).value == 7
