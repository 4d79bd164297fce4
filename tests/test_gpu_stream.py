"""The binding's default stream is torch's current stream of the current
device, whatever stream that is at the time of the call (GPU)."""
import pytest
import torch

from paper_2606_03026_gb300 import spikeproj as sp

pytestmark = pytest.mark.gpu


def test_default_stream_follows_torch():
    """Default stream, a side stream, nested side streams, and back; an explicit
    stream object or handle is taken as it is."""
    want = torch.cuda.default_stream().cuda_stream
    assert sp._stream(None) == want
    assert sp._stream(None) == want                      # the first call and the ones after it
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    with torch.cuda.stream(a):
        assert sp._stream(None) == a.cuda_stream
        with torch.cuda.stream(b):
            assert sp._stream(None) == b.cuda_stream == torch.cuda.current_stream().cuda_stream
        assert sp._stream(None) == a.cuda_stream
        assert sp._stream(b) == b.cuda_stream
        assert sp._stream(b.cuda_stream) == b.cuda_stream
    assert sp._stream(None) == want
