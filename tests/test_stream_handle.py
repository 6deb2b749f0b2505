"""The stream handle that a wrapper passes on, with fakes of torch's two ways to ask
for the current stream (no GPU)."""
from types import SimpleNamespace

import pytest
import torch

from paper_2605_13600_gb300 import scoup


@pytest.mark.parametrize("raw,initialized,want", [(True, True, 71), (True, False, 72), (False, True, 72), (False, False, 72)])
def test_current_stream(monkeypatch, raw, initialized, want):
    if raw:
        monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 70 + device, raising=False)
    else:
        monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "is_initialized", lambda: initialized)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 1)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: SimpleNamespace(cuda_stream=72))
    assert scoup._stream(None) == want


def test_given_stream():
    assert scoup._stream(SimpleNamespace(cuda_stream=5)) == 5
    assert scoup._stream(7) == 7 and scoup._stream(0) == 0
