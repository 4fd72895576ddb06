"""Edges of the record builders: columns of tilted cameras (32 samples at a time), level and tilted cameras in one rig, and the
feature copies of planar and ragged tensors, against the oracle."""
import numpy as np
import pytest

from paper_2607_10071_b200 import binding as fb
from paper_2607_10071_b200 import workloads as wl
from tests import parity
from tests.test_gpu_backward import check as check_backward

pytestmark = pytest.mark.gpu


def inputs(Z, mixed, N=3, C=16, dtype="f32", feat=(12, 17), grid=(11, 9)):
    w = wl.Workload("samples", 9000 + Z, 1, N, C, dtype, feat, (feat[0] * 8, feat[1] * 8), grid + (Z,),
                    (-6.0, 6.0, -6.0, 6.0, -3.0, 3.0), 0, general_pose=True)
    inp = wl.make_inputs(w)
    if mixed:  # every second camera without pitch and roll
        inp.lidar2img[:, ::2] = wl.ring_rig(N, 70.0, w.img_hw, np.full((1, N), 0.0173))[:, ::2]
    return inp


@pytest.mark.parametrize("mixed", [False, True])
@pytest.mark.parametrize("Z,slots16", [(1, 0), (2, 4), (31, 4), (32, 0), (33, 4), (65, 8), (200, 4), (300, 0)])
def test_samples_of_tilted_cameras(oracle, Z, slots16, mixed):
    inp = inputs(Z, mixed)
    w = inp.workload
    for reduce in (0, 1, 2):
        ref = oracle.sampling_vt(inp.features, inp.lidar2img, w.img_hw, w.bev_range, w.grid, reduce)
        out, cnt, _ = parity.run_gpu(inp, reduce, fb.KERNEL_TILED, (0, 0, 0, slots16 << 20))
        parity.assert_parity(w, ref, out, cnt, f"[Z={Z} reduce={reduce}]", check_fraction=False, large_outputs=True)
    check_backward(oracle, w, inp.lidar2img, 2, tune=(0, 0, 0, slots16 << 20))


@pytest.mark.parametrize("layout,dtype,C,feat", [
    (fb.NCHW, "f32", 4, (1, 1)), (fb.NCHW, "f32", 20, (5, 7)), (fb.NCHW, "f32", 36, (8, 32)), (fb.NCHW, "bf16", 8, (3, 3)),
    (fb.NCHW, "bf16", 72, (8, 64)), (fb.NCHW, "f32", 3, (1, 1)), (fb.NCHW, "f32", 33, (8, 32)), (fb.NCHW, "bf16", 9, (9, 57)),
    (fb.NCHW, "bf16", 35, (8, 8)), (fb.NCHW, "bf16", 40, (9, 57)), (fb.NHWC, "f32", 3, (1, 1)), (fb.NHWC, "f32", 9, (5, 7)),
    (fb.NHWC, "bf16", 9, (3, 3)), (fb.NHWC, "bf16", 33, (8, 31))])
def test_feature_copies(layout, dtype, C, feat):
    """The copy does not change a result: the same tensor through the caller's layout and as channels-last vectors."""
    import torch
    inp = inputs(9, True, C=C, dtype=dtype, feat=feat, grid=(39, 37))  # (planar tensors are padded from 12288 bins on)
    w = inp.workload
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    f = torch.from_numpy(inp.features).cuda().to(t)
    m = torch.from_numpy(inp.lidar2img).cuda()
    pad = -C % (8 if dtype == "bf16" else 4)
    ref = fb.sampling_vt(torch.nn.functional.pad(f, (0, pad)).contiguous(), m, w.img_hw, w.bev_range, w.grid)[..., :C]
    src = f.permute(0, 1, 4, 2, 3).contiguous() if layout == fb.NCHW else f
    out = fb.sampling_vt(src, m, w.img_hw, w.bev_range, w.grid, layout=layout)
    assert fb.flashbev_last_kernel_name().endswith("nchw" if layout == fb.NCHW else "padded")
    out = out.permute(0, 2, 3, 1) if layout == fb.NCHW else out
    # (planar tensors are worked on in other blocks of cells, so sums of tilted cameras' samples may be ordered differently)
    assert torch.equal(out, ref) or (layout == fb.NCHW and float((out - ref).abs().max()) <= 1e-5 * max(1.0, float(ref.abs().max())))


@pytest.mark.parametrize("C", [80, 84, 88, 96, 100, 128, 132, 144, 160, 192, 196])
def test_vectors_per_lane(oracle, C):
    """Channel counts on both sides of every change in the number of channel vectors per lane (fp32)."""
    inp = inputs(6, True, C=C)
    w = inp.workload
    for reduce in (0, 1):
        ref = oracle.sampling_vt(inp.features, inp.lidar2img, w.img_hw, w.bev_range, w.grid, reduce)
        out, cnt, _ = parity.run_gpu(inp, reduce, fb.KERNEL_TILED)
        parity.assert_parity(w, ref, out, cnt, f"[C={C} reduce={reduce}]", check_fraction=False)
    check_backward(oracle, w, inp.lidar2img, 0)
