"""The stream the binding hands to the library is torch's current one: it reads
it by torch's own low-level getters, which this pins to the public call."""
import pytest

from helpers import ensure_built


def test_the_getters_exist():
    import torch
    assert callable(torch._C._cuda_getCurrentRawStream) and callable(torch._C._cuda_getDevice)


@pytest.mark.gpu
def test_the_current_stream_is_used():
    ensure_built()
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2606_06510_gb300 as oz
    assert oz._stream() == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert oz._stream() == torch.cuda.current_stream().cuda_stream == side.cuda_stream
    assert oz._stream(side) == side.cuda_stream
