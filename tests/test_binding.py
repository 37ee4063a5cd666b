"""Host logic of the ctypes binding that needs no GPU."""
import torch

import paper_2512_08537_b200 as ardiff


class _Stream:
    def __init__(self, handle):
        self.cuda_stream = handle


def test_the_current_stream_with_and_without_torchs_number_of_it(monkeypatch):
    """torch's handle of the current stream as a number is not a public name: where it is missing the Stream object is asked."""
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 3)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: _Stream(77))
    monkeypatch.setattr(torch._C, "_cuda_getCurrentRawStream", lambda device: 1000 + device, raising=False)
    assert ardiff._stream_ptr(None) == 1003 and ardiff._stream_ptr(_Stream(5)) == 5
    monkeypatch.delattr(torch._C, "_cuda_getCurrentRawStream")
    assert ardiff._stream_ptr(None) == 77
