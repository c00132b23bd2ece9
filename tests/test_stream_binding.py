"""The binding's default stream is torch's current stream."""
import pytest

from gpu_common import load_pkg, need_gpu


@pytest.mark.gpu
def test_default_stream_follows_torch():
    torch = need_gpu()
    sp = load_pkg()
    assert sp._stream(None).value == (torch.cuda.current_stream().cuda_stream or None)
    st = torch.cuda.Stream()
    with torch.cuda.stream(st):
        assert sp._stream(None).value == st.cuda_stream
    assert sp._stream(st).value == st.cuda_stream
