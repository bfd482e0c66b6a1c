"""Parts of the session module that need no GPU."""
import importlib

import torch

from paper_2607_11136_b200 import session


def test_private_accessors_of_torch_have_public_stand_ins(monkeypatch):
    """Current device and stream come from torch's public functions where it lacks the direct ones."""
    try:
        with monkeypatch.context() as m:
            m.delattr(torch._C, "_cuda_getDevice")
            m.delattr(torch._C, "_cuda_getCurrentRawStream")
            m.setattr(torch.cuda, "current_stream", lambda index: type("Stream", (), {"cuda_stream": 40 + index}))
            importlib.reload(session)
            assert session._current_device is torch.cuda.current_device
            assert session._current_raw_stream(2) == 42
    finally:
        importlib.reload(session)
    assert session._current_raw_stream is torch._C._cuda_getCurrentRawStream
