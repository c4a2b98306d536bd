"""The stream a call without a stream argument launches on is torch's current one."""
import threading

import pytest
import torch

from paper_1909_11873_gb300 import gwl

pytestmark = pytest.mark.gpu


def test_default_stream_is_the_current_one():
    assert gwl._stream(None) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    seen = []
    with torch.cuda.stream(side):
        assert gwl._stream(None) == side.cuda_stream
        t = threading.Thread(target=lambda: seen.append(gwl._stream(None)))
        t.start()
        t.join()
    assert seen == [torch.cuda.default_stream().cuda_stream]   # the current stream is the thread's own
    assert gwl._stream(None) == torch.cuda.current_stream().cuda_stream
    ext = torch.cuda.ExternalStream(side.cuda_stream)
    with torch.cuda.stream(ext):
        assert gwl._stream(None) == side.cuda_stream


def test_default_stream_under_capture():
    x = torch.zeros(8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):
        assert gwl._stream(None) == torch.cuda.current_stream().cuda_stream
        x.add_(1.0)
    g.replay()
    torch.cuda.synchronize()
    assert float(x.sum()) == 8.0
