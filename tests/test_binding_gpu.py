"""The binding's argument marshalling on the GPU."""
import pytest

pytestmark = pytest.mark.gpu


def test_default_stream_is_the_current_one():
    """Calls without a stream go to the current device's current stream."""
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2605_29663_gb300 as ex
    assert ex._stream(None) == torch.cuda.current_stream().cuda_stream
    for s in (torch.cuda.Stream(), torch.cuda.Stream(priority=-1)):
        assert ex._stream(s) == s.cuda_stream
        with torch.cuda.stream(s):
            assert ex._stream(None) == s.cuda_stream
    assert ex._stream(None) == torch.cuda.current_stream().cuda_stream
