"""The current stream's handle in the Python binding: the same handle with and
without torch's internal call for it, and torch's own error where there is no
GPU."""
import pytest
import torch

from paper_2606_00724_gb300 import wf


@pytest.mark.skipif(torch.cuda.is_available(), reason="needs a machine without a GPU")
@pytest.mark.parametrize("internal", [True, False])
def test_no_gpu_raises_as_torch_does(monkeypatch, internal):
    if not internal:
        monkeypatch.setattr(wf, "_raw_stream", None)
    with pytest.raises(Exception) as want:
        torch.cuda.current_stream()
    with pytest.raises(type(want.value)):
        wf._stream(None)


@pytest.mark.gpu
def test_current_stream(monkeypatch):
    side = torch.cuda.Stream()
    for internal in (True, False):
        if not internal:
            monkeypatch.setattr(wf, "_raw_stream", None)
        assert wf._stream(None) == torch.cuda.current_stream().cuda_stream
        with torch.cuda.stream(side):
            assert wf._stream(None) == side.cuda_stream
        assert wf._stream(side) == side.cuda_stream
