"""The binding's default stream is the current one of the current device."""
import pytest

from paper_2406_06385_gb300 import lrqat as LQ

from gpu_util import torch

pytestmark = pytest.mark.gpu


def test_default_stream_is_the_current_one():
    t = torch()
    t.zeros(1, device="cuda")
    assert LQ._stream(None) == t.cuda.current_stream().cuda_stream
    side = t.cuda.Stream()
    with t.cuda.stream(side):
        assert LQ._stream(None) == side.cuda_stream
    assert LQ._stream(side) == side.cuda_stream
    assert LQ._stream(None) == t.cuda.current_stream().cuda_stream
