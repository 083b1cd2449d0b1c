"""The binding's way to the current stream does not depend on functions that a torch release may drop."""
from types import SimpleNamespace

import torch

from paper_2501_07139_b200 import flexq


def test_stream_without_the_short_way(monkeypatch):
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: True)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: SimpleNamespace(cuda_stream=1234))
    for missing in ("_raw_stream", "_device"):
        with monkeypatch.context() as m:
            m.setattr(flexq, missing, None)
            assert flexq._stream() == 1234
    monkeypatch.setattr(flexq, "_device", lambda: 3)
    monkeypatch.setattr(flexq, "_raw_stream", lambda device: 100 + device)
    assert flexq._stream() == 103
