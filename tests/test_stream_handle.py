"""The binding's default stream handle does not depend on torch's internal function
for it (no GPU: torch's calls are replaced)."""
import torch

from paper_2608_24348_gb300 import sem


class _Stream:
    cuda_stream = 1234


def test_stream_handle_without_the_internal_function(monkeypatch):
    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: _Stream())
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    assert sem.stream_ptr() == 1234
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda d: 5678 + d, raising=False)
    assert sem.stream_ptr() == 5678
    assert sem.stream_ptr(_Stream()) == 1234
