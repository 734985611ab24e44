"""A call without a stream runs on the caller's current stream."""
import threading

import pytest

import paper_2111_06906_gb300 as pv

pytestmark = pytest.mark.gpu


def test_default_is_the_current_stream():
    import torch
    side = torch.cuda.Stream()
    seen = {}

    def other_thread():
        seen["thread"] = pv._stream(None).value

    assert (pv._stream(None).value or 0) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert pv._stream(None).value == side.cuda_stream
        t = threading.Thread(target=other_thread)      # the current stream is each thread's own
        t.start()
        t.join()
    assert (seen["thread"] or 0) == torch.cuda.default_stream().cuda_stream
    assert (pv._stream(None).value or 0) == torch.cuda.current_stream().cuda_stream
