"""The binding's default stream is PyTorch's current one: on the default stream, inside a stream
context, back outside it, and in another thread (whose current stream is its own)."""
import threading

import pytest
import torch

from paper_2604_10044_gb300 import lg

pytestmark = pytest.mark.gpu


def _agrees():
    return lg._stream(None) == torch.cuda.current_stream().cuda_stream


def test_default_stream_is_the_current_one(cuda):
    torch.zeros(1, device=cuda)
    side = torch.cuda.Stream(device=cuda)
    assert _agrees()
    with torch.cuda.stream(side):
        assert lg._stream(None) == side.cuda_stream
        seen = []
        other = threading.Thread(target=lambda: seen.append((_agrees(), lg._stream(None))))
        other.start()
        other.join()
        assert seen[0][0] and seen[0][1] != side.cuda_stream
    assert _agrees()
    assert lg._stream(side) == side.cuda_stream and lg._stream(12345) == 12345
