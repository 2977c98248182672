"""The stream that a call runs on: the current one of the calling thread, or
the one that is passed."""
import threading

import pytest
import torch

pytestmark = pytest.mark.gpu


def test_stream_argument():
    from paper_2405_16406_gb300 import spinq as S
    s, t = torch.cuda.Stream(), torch.cuda.Stream()
    assert S._stream(None) == torch.cuda.current_stream().cuda_stream
    assert S._stream(s) == s.cuda_stream
    seen = []
    with torch.cuda.stream(s):
        assert S._stream(None) == s.cuda_stream and S._stream(t) == t.cuda_stream
        th = threading.Thread(target=lambda: seen.append(S._stream(None)))
        th.start()
        th.join()
    assert seen == [torch.cuda.default_stream().cuda_stream]
    assert S._stream(None) == torch.cuda.current_stream().cuda_stream
