"""The handle of the current stream, which every call is made with: from torch's private function where there is one, else through the public object."""
import pytest
import torch

from paper_2602_01801_b200 import fastar


def test_without_the_private_function(monkeypatch):
    monkeypatch.setattr(fastar, "_raw_stream", None)
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream", raising=False)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda device: type("Stream", (), dict(cuda_stream=1000 + device)))
    assert fastar._stream() == 1003


@pytest.mark.gpu
def test_it_is_the_current_stream():
    side = torch.cuda.Stream()
    assert fastar._stream() == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert fastar._stream() == side.cuda_stream == torch.cuda.current_stream().cuda_stream
    assert fastar._stream() == torch.cuda.current_stream().cuda_stream
