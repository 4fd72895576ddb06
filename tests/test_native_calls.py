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
