"""The binding's default stream is torch's current stream of the current device, in every thread."""
import threading

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_default_stream_is_the_current_one():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0906_1887_gb300 import corr
    assert corr._stream_handle(None) == torch.cuda.current_stream().cuda_stream
    side = torch.cuda.Stream()
    seen = []
    with torch.cuda.stream(side):
        assert corr._stream_handle(None) == side.cuda_stream != 0
        th = threading.Thread(target=lambda: seen.append(corr._stream_handle(None)))   # its own current stream
        th.start()
        th.join()
    assert seen == [torch.cuda.default_stream().cuda_stream]
    assert corr._stream_handle(None) == torch.cuda.current_stream().cuda_stream
