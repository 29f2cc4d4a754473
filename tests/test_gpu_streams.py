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


def scene_plan(sar, n_range, n_az, seed):
    return sar.sar_plan_create(n_range, n_az, randn(n_range, seed=seed), randn(n_az, seed=seed + 1))


# every kind of launch behind a predecessor: the latency kernels, folds in clusters and through tensor stores,
# mixed radix, zero-padded lengths with corner turns; the last scene's passes are too large and launched ordinarily
SCENES = [(256, 256), (1024, 256), (4096, 64), (2048, 608), (1000, 300), (1021, 333), (4096, 4096), (4096, 8192)]


@pytest.mark.parametrize("n_range,n_az", SCENES)
def test_scene_behind_captured_copies_and_joined_streams(sar, n_range, n_az):
    """Captured behind a memset and a copy node, behind two streams that join, and before a copy node: every
    replay reads what the nodes before it wrote and is complete for those after it."""
    plan = scene_plan(sar, n_range, n_az, 3)
    a, b = randn(n_az, n_range, seed=5), randn(n_az, n_range, seed=6)
    empty = lambda: torch.empty((n_range, n_az), dtype=torch.complex64, device="cuda")
    work, side_work, image, side_image, last = empty(), empty(), empty(), empty(), empty()
    raw, side_raw, both = torch.empty_like(a), torch.empty_like(a), torch.empty_like(a)
    side, copied = torch.cuda.Stream(), empty()

    def wanted(x):
        sar.sar_rda_process_oop(plan, x, work, image)
        torch.cuda.synchronize()
        return image.clone()
    wanted(a)
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        raw.zero_()
        raw.copy_(a)
        sar.sar_rda_process_oop(plan, raw, work, image)                   # behind a copy node
        here = torch.cuda.current_stream()
        side.wait_stream(here)
        with torch.cuda.stream(side):
            side_raw.copy_(b)
            sar.sar_rda_process_oop(plan, side_raw, side_work, side_image)
        copied.copy_(image)                                               # behind the scene's last kernel
        sar.sar_rda_process_oop(plan, a, work, image)
        here.wait_stream(side)
        both.view(n_range, n_az).copy_(image + side_image)
        sar.sar_rda_process_oop(plan, both, work, last)                   # behind kernels of two streams
    for _ in range(3):
        for x in (a, b):
            x.copy_(x.roll(1, 0))
        for x in (raw, side_raw, both, image, side_image, copied, last):
            x.fill_(float("nan"))
        graph.replay()
        torch.cuda.synchronize()
        got = [copied.clone(), side_image.clone(), last.clone()]
        first, second = wanted(a), wanted(b)
        total = (first + second).view(n_az, n_range).clone()
        for g, w in zip(got, (first, second, wanted(total))):
            assert torch.equal(g, w)
    plan.destroy()


@pytest.mark.parametrize("n_range,n_az", SCENES)
def test_two_plans_alternate_on_two_streams(sar, n_range, n_az):
    """Each stream's scene waits, by an event of the caller, for the echo that the other stream is still
    making, and follows its own stream's last scene directly: as one after the other on one stream."""
    plans = [scene_plan(sar, n_range, n_az, 11), scene_plan(sar, n_range, n_az, 13)]
    empty = lambda: torch.empty((n_range, n_az), dtype=torch.complex64, device="cuda")
    start = randn(n_az, n_range, seed=15)
    rounds = 6

    def go(streams):
        raws = [start.clone()] + [torch.empty_like(start) for _ in range(rounds)]
        images, works = [empty() for _ in range(rounds)], [empty() for _ in range(2)]
        torch.cuda.synchronize()
        ready = torch.cuda.Event()
        ready.record(streams[0])
        for k in range(rounds):
            with torch.cuda.stream(streams[k % 2]):
                streams[k % 2].wait_event(ready)
                sar.sar_rda_process_oop(plans[k % 2], raws[k], works[k % 2], images[k])
                ready = torch.cuda.Event()
                raws[k + 1].view(n_range, n_az).copy_(images[k])
                ready.record()
                # more of the library's work on this stream, for the next scene here to be launched behind
                sar.sar_rda_process_oop(plans[k % 2], start, works[k % 2], works[k % 2].new_empty((n_range, n_az)))
        torch.cuda.synchronize()
        return images
    want = go([torch.cuda.current_stream()] * 2)
    for _ in range(3):
        for g, w in zip(go([torch.cuda.Stream(), torch.cuda.Stream()]), want):
            assert torch.equal(g, w)
    for p in plans:
        p.destroy()
