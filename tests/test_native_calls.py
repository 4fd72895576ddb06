"""The functions for torch tensors (``sampling_vt`` and the like) as ordinary citizens of a PyTorch program: the errors they
raise, the threads and streams they share the process with."""
import pytest

from paper_2607_10071_b200 import binding as fb

RANGE = (-10.0, 10.0, -10.0, 10.0, -3.0, 2.0)


def _fake_cuda(*shape):
    """A CUDA tensor without memory, which exists on machines without a GPU too."""
    torch = pytest.importorskip("torch")
    from torch._subclasses.fake_tensor import FakeTensorMode
    with FakeTensorMode():
        return torch.empty(shape, device="cuda")


def test_rig_with_too_few_dimensions_is_an_index_error():
    grad, rig = _fake_cuda(1, 5, 6, 8), _fake_cuda(4)
    with pytest.raises(IndexError):
        fb.sampling_vt_backward(grad, rig, (8, 8), (64, 64), RANGE, (5, 6, 4))


def test_backward_refuses_a_rig_that_its_kernel_cannot_read():
    """As the other calls do: host memory, other number types, strides."""
    torch = pytest.importorskip("torch")
    grad, rig = _fake_cuda(1, 5, 6, 8), _fake_cuda(1, 2, 4, 4)
    for bad in (torch.zeros((1, 2, 4, 4)), rig.to(torch.float64), rig.transpose(2, 3)):
        with pytest.raises(ValueError, match="lidar2img"):
            fb.sampling_vt_backward(grad, bad, (8, 8), (64, 64), RANGE, (5, 6, 4))


@pytest.mark.gpu
def test_numbers_are_converted_as_python_converts_them():
    """bev_range by float(), hints by int(), level_hw as numpy casts it; the backward reads the height bins only from the grid."""
    import numpy as np
    import torch
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(3)
    f = torch.randn((1, 2, 4, 6, 8), generator=gen, device=dev)
    m = torch.eye(4, device=dev).expand(1, 2, 4, 4).contiguous()
    m[:, :, :3, 3] = torch.tensor([24.0, 16.0, 4.0], device=dev)
    img, r, grid = (32, 48), (-1.0, 1.0, -1.0, 1.0, -1.0, 1.0), (5, 6, 4)
    want = fb.sampling_vt(f, m, img, r, grid)
    assert float(want.abs().sum()) > 0
    for ranges in (np.asarray(r, np.float32), torch.tensor(r), [str(v) for v in r]):
        assert torch.equal(fb.sampling_vt(f, m, np.asarray(img), ranges, torch.tensor(grid), tune=(0.0, 0.0, np.float32(0), 0)), want)
    grad = torch.randn((1, 5, 6, 8), generator=gen, device=dev)
    back = fb.sampling_vt_backward(grad, m, (4, 6), img, r, grid)
    assert torch.allclose(fb.sampling_vt_backward(grad, m, (4, 6), img, r, (None, None, 4, None)), back, rtol=1e-5, atol=1e-5)
    value = torch.randn((1, 2, 30, 2, 8), generator=gen, device=dev)
    off = torch.randn((1, 30, 2, 2, 4, 2), generator=gen, device=dev)
    wts = torch.rand((1, 30, 2, 2, 4), generator=gen, device=dev)
    att = fb.sca(value, ((4, 6), (2, 3)), m, off, wts, img, r, grid)
    for hw in (np.array([[4, 6], [2, 3]]), np.array([4.0, 6.0, 2.0, 3.0]), torch.tensor([[4, 6], [2, 3]]), [4, 6, 2, 3, 9, 9],
               torch.tensor([4.5, 6.0, 2.0, 3.0]), [[4, 6], np.array([2, 3])]):
        assert torch.equal(fb.sca(value, hw, m, off, wts, img, r, grid, chunk_records=0.0), att)
    with pytest.raises(ValueError):
        fb.sca(value, [4, 6, 2], m, off, wts, img, r, grid)


@pytest.mark.gpu
def test_failed_allocation_is_an_out_of_memory_error_and_leaves_the_device_usable():
    import torch
    dev = torch.device("cuda:0")
    f, m = torch.ones((1, 2, 4, 6, 512), device=dev), torch.eye(4, device=dev).expand(1, 2, 4, 4).contiguous()
    geo = ((32, 48), RANGE)
    huge = 40000                                   # 40000 x 40000 rows of 512 floats: 3.3 TB
    calls = [lambda: fb.sampling_vt(f, m, *geo, (huge, huge, 1)),
             lambda: fb.sampling_vt_multires([f], m, *geo, (huge, huge, 1)),
             lambda: fb.sampling_vt_backward(torch.ones((1, 4, 4, 512), device=dev), m, (huge, huge), *geo, (4, 4, 1)),
             lambda: fb.sca(torch.ones((1, 2, 24, 8, 64), device=dev), ((4, 6),), m, torch.zeros((1, 16, 8, 1, 4, 2), device=dev),
                            torch.ones((1, 16, 8, 1, 4), device=dev), *geo, (huge, huge, 1))]
    for call in calls:
        with pytest.raises(torch.OutOfMemoryError):
            call()
    out = fb.sampling_vt(f, m, *geo, (4, 4, 1))
    torch.cuda.synchronize()
    assert out.shape == (1, 4, 4, 512) and bool(torch.isfinite(out).all())


@pytest.mark.gpu
def test_other_threads_run_while_a_call_waits():
    """A call that finds the stream's launch queue full waits for room in it, without the interpreter lock."""
    import threading
    import time

    import torch
    dev = torch.device("cuda:0")
    f, m = torch.ones((1, 2, 4, 6, 8), device=dev), torch.eye(4, device=dev).expand(1, 2, 4, 4).contiguous()
    out = torch.empty((1, 4, 4, 8), device=dev)
    fb.sampling_vt(f, m, (32, 48), RANGE, (4, 4, 1), out=out)
    torch.cuda.synchronize()
    ticks, stop = [], threading.Event()

    def tick():
        while not stop.is_set():
            ticks.append(time.perf_counter())
            time.sleep(0.001)

    thread = threading.Thread(target=tick)
    thread.start()
    try:
        torch.cuda._sleep(1_000_000_000)           # half a second of an idle GPU at the head of the stream
        longest = (0.0, 0.0)
        for _ in range(20000):
            t0 = time.perf_counter()
            fb.sampling_vt(f, m, (32, 48), RANGE, (4, 4, 1), out=out)
            longest = max(longest, (time.perf_counter() - t0, t0))
            if longest[0] > 0.1:
                break
        torch.cuda.synchronize()
    finally:
        stop.set()
        thread.join()
    waited, since = longest
    assert waited > 0.1, "no call had to wait"
    during = [t for t in ticks if since < t < since + waited]
    gaps = [b - a for a, b in zip([since] + during, during + [since + waited])]
    assert max(gaps) < 0.5 * waited, f"the other thread stood still for {max(gaps):.3f} s of a wait of {waited:.3f} s"


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["planar", "ragged", "pyramid"])
def test_memory_of_a_call_on_a_named_stream_belongs_to_that_stream(call):
    """Scratch and result come from the named stream's memory: what is allocated later for another stream never gets the scratch
    while the call may still use it, and a dropped result is not handed out again while the caller's stream may still read it."""
    import torch
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(5)
    m = torch.eye(4, device=dev).expand(1, 2, 4, 4).contiguous()
    m[:, :, :3, 3] = torch.tensor([24.0, 16.0, 4.0], device=dev)
    img, r, grid = (32, 48), (-1.0, 1.0, -1.0, 1.0, -1.0, 1.0), (90, 90, 4)
    C = 30 if call == "ragged" else 32
    shape = (1, 2, 120, 170, C) if call == "ragged" else (1, 2, C, 120, 170)
    f = torch.randn(shape, generator=gen, device=dev)
    layout = fb.NHWC if call == "ragged" else fb.NCHW

    def run(**kw):
        if call == "pyramid":
            return fb.sampling_vt_multires([f, f], m, img, r, grid, layout=layout, **kw)
        return fb.sampling_vt(f, m, img, r, grid, layout=layout, **kw)

    want = run()
    assert fb.flashbev_last_kernel_name().startswith("tiled")
    side = torch.cuda.Stream()
    out = torch.empty_like(want)
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    before = {s["address"] for s in torch.cuda.memory_snapshot()}
    run(out=out, stream=side.cuda_stream)
    fresh = [s for s in torch.cuda.memory_snapshot() if s["address"] not in before]
    scratch = 2 * 120 * 170 * 32 * 4
    assert sum(s["total_size"] for s in fresh) >= scratch, "the scratch was not allocated in this call"
    assert {s["stream"] for s in fresh} == {side.cuda_stream}
    side.synchronize()
    assert torch.equal(out, want)
    # a result of the call: the named stream's memory, kept while the caller's stream still works with it
    res = run(stream=side.cuda_stream)
    where = res.data_ptr()
    assert any(s["address"] <= where < s["address"] + s["total_size"] for s in torch.cuda.memory_snapshot()
               if s["stream"] == side.cuda_stream)
    torch.cuda.current_stream().wait_stream(side)
    torch.cuda._sleep(200_000_000)
    copy = res.clone()
    del res
    again = run(stream=side.cuda_stream)
    assert again.data_ptr() != where
    torch.cuda.synchronize()
    assert torch.equal(copy, want) and torch.equal(again, want)


@pytest.mark.gpu
def test_default_stream_handles():
    import torch
    dev = torch.device("cuda:0")
    f, m = torch.ones((1, 2, 4, 6, 8), device=dev), torch.eye(4, device=dev).expand(1, 2, 4, 4).contiguous()
    want = fb.sampling_vt(f, m, (32, 48), RANGE, (4, 4, 1))
    for handle in (0, 1, 2):                       # NULL, the legacy stream's and the per-thread stream's own handles
        got = fb.sampling_vt(f, m, (32, 48), RANGE, (4, 4, 1), stream=handle)
        torch.cuda.synchronize()
        assert torch.equal(got, want)
