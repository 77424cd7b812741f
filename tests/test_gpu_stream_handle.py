"""The binding's current-stream handle is torch's current stream's."""
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_current_stream_handle():
    from paper_2606_26547_gb300 import hdc
    torch.zeros(1, device="cuda")
    handle = lambda: hdc._stream().value or 0
    assert handle() == torch.cuda.current_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert handle() == s.cuda_stream == (hdc._stream(s).value or 0)
    assert handle() == torch.cuda.current_stream().cuda_stream
