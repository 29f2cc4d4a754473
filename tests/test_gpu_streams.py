"""GPU: the library's launches among the caller's own work on streams."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def sar(built_lib):
    import paper_2604_03585_gb300 as sar
    assert torch.cuda.is_available(), "gpu tests need a CUDA device"
    torch.cuda.set_device(0)
    return sar


def randn(*shape, seed=0):
    return torch.randn(shape, dtype=torch.complex64, device="cuda", generator=torch.Generator("cuda").manual_seed(seed))


@pytest.mark.parametrize("n", [1024, 32768], ids=["one_block", "cluster"])
def test_refused_launch_leaves_no_error_for_the_next_call(sar, n):
    """A launch into a capture that has become invalid is refused by the host; the next call, on another
    stream, is not told of it."""
    x, y = randn(4, n), torch.empty((4, n), dtype=torch.complex64, device="cuda")
    prime = randn(4, 1021, seed=1)
    got = torch.empty_like(prime)
    sar.sar_fft_lines(n, 4, x, y)                       # tables of both lengths
    sar.sar_fft_lines(1021, 4, prime, got)
    want = got.clone()
    torch.cuda.synchronize()
    runtime = ctypes.CDLL("libcudart.so.13")            # torch's; the library has one of its own
    stream = torch.cuda.Stream()
    handle, graph = ctypes.c_void_p(stream.cuda_stream), ctypes.c_void_p()
    assert runtime.cudaStreamBeginCapture(handle, 2) == 0             # relaxed mode
    assert runtime.cudaStreamSynchronize(handle) != 0                 # not allowed there: the capture is invalid
    with pytest.raises(sar.SarError) as e:
        sar.sar_fft_lines(n, 4, x, y, stream=stream)
    assert e.value.status == sar.SAR_ERR_CUDA
    assert runtime.cudaStreamEndCapture(handle, ctypes.byref(graph)) != 0
    runtime.cudaGetLastError()
    got.zero_()
    sar.sar_fft_lines(1021, 4, prime, got)
    assert torch.equal(got, want)
