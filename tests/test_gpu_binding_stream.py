"""The binding launches on torch's current stream of the current device, whichever that is at the call."""

import threading

import pytest

from paper_2605_28451_gb300 import bfpfft as B

pytestmark = pytest.mark.gpu


def test_current_stream_is_followed(cuda_ready):
    import torch

    def same():
        return B._stream(None) == torch.cuda.current_stream().cuda_stream
    assert same()
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(first):
        assert same() and B._stream(None) == first.cuda_stream
        with torch.cuda.stream(second):
            assert same() and B._stream(None) == second.cuda_stream
        assert B._stream(None) == first.cuda_stream
    seen = []
    t = threading.Thread(target=lambda: seen.append((B._stream(None), torch.cuda.current_stream().cuda_stream)))
    with torch.cuda.stream(first):
        t.start()
        t.join()                                  # another thread has its own current stream
    assert seen[0][0] == seen[0][1]
    assert B._stream(first) == first.cuda_stream and B._stream(17) == 17
