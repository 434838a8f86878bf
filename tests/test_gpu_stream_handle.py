"""The stream a call runs on by default is the current one, in and out of a stream context."""
import pytest
import torch

from paper_2604_09884_gb300 import inrct

pytestmark = pytest.mark.gpu


def test_default_stream_is_the_current_one():
    torch.zeros(1, device="cuda")
    for ctx in (torch.cuda.Stream(), torch.cuda.default_stream(), torch.cuda.Stream(priority=-1)):
        with torch.cuda.stream(ctx):
            assert (inrct._stream().value or 0) == torch.cuda.current_stream().cuda_stream == ctx.cuda_stream
    assert inrct._stream(ctx).value == ctx.cuda_stream
