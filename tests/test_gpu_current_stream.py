"""The binding's default stream is torch's current one, whatever it is."""
import pytest

pytestmark = pytest.mark.gpu


def test_default_stream_is_torchs_current_stream():
    import torch

    from paper_2501_01628_gb300 import vr
    assert (vr._stream(None).value or 0) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        assert vr._stream(None).value == side.cuda_stream
    assert (vr._stream(None).value or 0) == torch.cuda.default_stream().cuda_stream
