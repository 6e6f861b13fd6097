"""The stream handle of a call (CPU): an explicit stream's own, the current
stream's otherwise, also with a torch that has no raw-handle function."""
import types

import pytest
import torch

from paper_2407_18015_gb300 import ucp


def test_explicit_stream():
    assert ucp._stream(types.SimpleNamespace(cuda_stream=7), torch.device("cuda", 0)) == 7


@pytest.mark.parametrize("device", [None, torch.device("cuda"), torch.device("cuda", 1)])
def test_without_the_raw_handle(monkeypatch, device):
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    seen = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda d=None: (
        seen.append(d), types.SimpleNamespace(cuda_stream=11))[1])
    assert ucp._stream(None, device) == 11 and seen == [device]
