"""The stream a call runs on when none is given."""
from types import SimpleNamespace

import pytest
import torch

from paper_2609_22755_b200 import binding as B


@pytest.mark.parametrize("direct", [True, False])
def test_current_stream(monkeypatch, direct):
    """Its handle is asked for directly where torch has that call, and taken from the Stream object where it has not."""
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=0x1234))
    if direct:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 0x1230 + device, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert B._stream_ptr(None) == (0x1233 if direct else 0x1234)
    assert B._stream_ptr(0x77) == 0x77
    assert B._stream_ptr(SimpleNamespace(cuda_stream=0x88)) == 0x88
