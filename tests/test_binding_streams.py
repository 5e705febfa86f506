"""The binding's argument checks and the stream it launches on."""
import pytest

from paper_2609_38169_gb300 import api as A


def test_cpu_tensors_are_refused():
    torch = pytest.importorskip("torch")
    x = torch.zeros(2, 2, 4, 128)
    with pytest.raises(ValueError, match="expected a CUDA tensor"):
        A.stepq_prefill_fp32(A.Config(1, 4, 4), x, x, x, x, x, x, x)


@pytest.mark.gpu
def test_current_and_given_streams():
    torch = pytest.importorskip("torch")
    side = torch.cuda.Stream()
    assert A._stream(None) == torch.cuda.current_stream().cuda_stream
    with torch.cuda.stream(side):
        assert A._stream(None) == side.cuda_stream
    assert A._stream(side) == side.cuda_stream
    assert A._stream(None) == torch.cuda.current_stream().cuda_stream
    t = torch.zeros(4, 4, device="cuda")
    with pytest.raises(ValueError, match="contiguous"):
        A._dev_ptr(t.t()[1:])
    with pytest.raises(ValueError, match="expected torch.int32, got torch.float32"):
        A._dev_ptr(t, torch.int32)
    assert A._dev_ptr(None) is None and A._dev_ptr(t, torch.float32) == t.data_ptr()
