"""Calls without a stream go to torch's current stream, whichever that is at the call."""
import pytest

import paper_2609_07966_gb300 as mkv

from gpu_util import torch_cuda

pytestmark = pytest.mark.gpu


def test_default_is_the_current_stream():
    torch = torch_cuda()
    torch.cuda.init()
    assert mkv._stream(None) == torch.cuda.current_stream().cuda_stream
    for side in (torch.cuda.Stream(), torch.cuda.Stream(priority=-1)):
        with torch.cuda.stream(side):
            assert mkv._stream(None) == side.cuda_stream
            assert mkv._stream(0) == 0
    assert mkv._stream(None) == torch.cuda.current_stream().cuda_stream
