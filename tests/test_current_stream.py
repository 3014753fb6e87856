"""The binding's current stream with and without torch's raw-handle accessor."""
from types import SimpleNamespace

import pytest


@pytest.mark.parametrize("raw", [True, False])
def test_current_stream(monkeypatch, raw):
    import torch
    from paper_2609_03922_gb300 import spdba
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=17))
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 17 + d, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert spdba.current_stream() == (20 if raw else 17)
