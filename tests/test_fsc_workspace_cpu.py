"""The FSC's workspace is optional: a torch that cannot give one (no CUDA in
it, no driver, no room) leaves the allocation to the library."""
import pytest
import torch

from paper_1905_13408_gb300 import spg


class _Stream:
    cuda_stream = 0


@pytest.mark.parametrize("stream", [None, 0, 4096])
@pytest.mark.parametrize("error", [AssertionError("Torch not compiled with CUDA enabled"),
                                   RuntimeError("Found no NVIDIA driver on your system"),
                                   torch.cuda.OutOfMemoryError("out of memory")], ids=["no-cuda", "no-driver", "no-room"])
def test_no_workspace_from_torch(error, stream, monkeypatch):
    def fails(*a, **k):
        raise error

    if isinstance(error, torch.cuda.OutOfMemoryError):
        monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream())
        monkeypatch.setattr(torch, "empty", fails)
        monkeypatch.setattr(torch.cuda, "ExternalStream", lambda h: _Stream())
        monkeypatch.setattr(torch.cuda, "stream", lambda s: torch.no_grad())
    else:
        monkeypatch.setattr(torch.cuda, "current_stream", fails)
    assert spg._workspace(1024, stream) is None
