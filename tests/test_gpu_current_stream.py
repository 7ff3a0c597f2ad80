"""Which stream a call without one is enqueued on: the thread's current stream."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_calls_go_to_the_current_stream_of_the_thread():
    from paper_2609_04526_gb300 import _lib
    torch.zeros(1, device="cuda")
    side, other, seen = torch.cuda.Stream(), torch.cuda.Stream(), []

    def thread():
        seen.append(_lib._stream(None))   # a new thread starts on the default stream
        with torch.cuda.stream(other):
            seen.append(_lib._stream(None))

    assert _lib._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert _lib._stream(None) == side.cuda_stream
        t = threading.Thread(target=thread)
        t.start()
        t.join()
        assert _lib._stream(None) == side.cuda_stream
    assert seen == [torch.cuda.default_stream().cuda_stream, other.cuda_stream]
    assert _lib._stream(side) == _lib._stream(side.cuda_stream) == side.cuda_stream
