"""The stream that a call takes from its arrays (no GPU needed: the arrays and
torch's stream lookups are stand-ins)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

import paper_2608_21763_gb300 as s2w  # noqa: E402


class OnGpu:
    is_cuda, device = True, "cuda:3"

    def get_device(self):
        return 3


class Stream:
    cuda_stream = 77


def test_stream_of_the_arrays_with_and_without_torchs_raw_handle(monkeypatch):
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda i: 1000 + i, raising=False)
    assert s2w._stream(None, np.zeros(2), None, OnGpu()) == 1003
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    asked = []
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: asked.append(device) or Stream())
    assert s2w._stream(None, OnGpu()) == 77 and asked == ["cuda:3"]


def test_explicit_and_host_only_calls():
    assert s2w._stream(Stream(), OnGpu()) == 77 and s2w._stream(5, OnGpu()) == 5
    assert s2w._stream(None, np.zeros(2)) is None
