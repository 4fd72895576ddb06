"""Performance cases: the calls a user of this package makes, at the sizes they make them.

The view transformation runs once per frame inside a bird's-eye-view network, on the feature maps that the image
backbone left on the GPU: forward in serving and training, backward in training, its spatial cross-attention relative
(FlashSCA) in transformer models, and the sum over a feature pyramid.  Sizes are those of the package's workloads
(`workloads.py`, `bench.py`) and of its tests.  Half of the cases use rigs without pitch and roll (the benchmark's),
half use calibrated rigs, where every camera has its own pitch, roll, offset and focal length, as on a real vehicle.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_10071_b200 import binding as fb
from paper_2607_10071_b200 import workloads as wl

SUM, MEAN, EQ1 = fb.REDUCE_SUM, fb.REDUCE_MEAN_OVER_VALID, fb.REDUCE_CAMERA_MEAN_Z_SUM


def _vt(name, kind, **k):
    """A case of the sampling operator (`kind`: forward, backward or pyramid)."""
    c = dict(name=name, kind=kind, B=1, N=6, C=80, dtype="f32", out="f32", layout="nhwc", Hf=32, Wf=88, Himg=256, Wimg=704,
             X=200, Y=200, Z=8, xy=50.0, z0=-5.0, z1=3.0, reduce=SUM, rig="level", fov=70.0, levels=1, count=False)
    c.update(k)
    return c


def _sca(name, **k):
    """A case of the spatial cross-attention."""
    c = dict(name=name, kind="sca", B=1, N=6, heads=8, Dh=32, dtype="f32", L=4, P=8, Himg=928, Wimg=1600, stride=8,
             X=200, Y=200, Zref=4, xy=51.2, z0=-5.0, z1=3.0, rig="level")
    c.update(k)
    return c


def listed():
    return [
        # the smallest call: a coarse grid for a low-speed or parking function, bound by latency and by the host's work
        _vt("tiny", "forward", C=32, Hf=16, Wf=44, Himg=128, Wimg=352, X=50, Y=50, Z=4, xy=25.0, z0=-3.0, z1=1.0),
        # the ordinary call: six cameras, stride-8 maps, a 0.5 m grid of 100 m by 100 m, single precision
        _vt("representative", "forward"),
        # the paper's own shape and reduction (mean over cameras, sum over heights) on a calibrated rig
        _vt("paper_calibrated", "forward", C=128, Hf=56, Wf=100, Himg=448, Wimg=800, z1=5.0, reduce=EQ1, rig="calibrated"),
        # two frames in one call, half-precision maps, mean over the valid samples, the counts wanted as well
        _vt("half_taller", "forward", B=2, C=128, dtype="bf16", Z=16, reduce=MEAN, count=True),
        # a 200 m by 200 m grid over stride-4 maps
        _vt("long_range", "forward", C=128, dtype="bf16", Hf=64, Wf=176, X=400, Y=400, Z=16, xy=100.0),
        # 0.2 m cells and 64 height bins (occupancy), eight cameras
        _vt("high_res", "forward", N=8, C=64, dtype="bf16", Hf=64, Wf=176, X=512, Y=512, Z=64, xy=51.2, fov=60.0),
        # channel planes in and out, as convolutional networks keep them, bf16 throughout, calibrated cameras
        _vt("planar_calibrated", "forward", C=128, dtype="bf16", out="bf16", layout="nchw", Hf=64, Wf=176, Z=16, rig="calibrated"),
        # nothing divides anything: odd map, odd grid, a channel count that is no multiple of four
        _vt("ragged", "forward", N=5, C=82, Hf=29, Wf=77, Himg=232, Wimg=616, X=181, Y=203, Z=11, rig="calibrated"),
        # training: the gradient with respect to the features
        _vt("backward", "backward"),
        _vt("backward_calibrated", "backward", C=128, Hf=56, Wf=100, Himg=448, Wimg=800, z1=5.0, reduce=EQ1, rig="calibrated"),
        # strides 8, 16 and 32 of a feature pyramid summed into one grid
        _vt("pyramid", "pyramid", C=128, dtype="bf16", Z=16, levels=3),
        # spatial cross-attention at BEVFormer-base sizes
        _sca("sca"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


#: What no drawn call exceeds: the largest listed ones.
_MOST_SAMPLES, _MOST_OUT = 512 * 512 * 64 * 64, 400 * 400 * 128


def draw(rng):
    """One more call: sizes over the whole range of the listed ones, odd ones among them."""
    kind = rng.choices(("forward", "backward", "pyramid", "sca"), (55, 20, 12, 13))[0]
    rig = rng.choice(("level", "calibrated"))
    if kind == "sca":
        c = _sca("", dtype=rng.choice(("f32", "bf16")), L=rng.choice((1, 2, 3, 4)), P=rng.choice((4, 8)), N=rng.choice((4, 5, 6)),
                 X=_log_int(rng, 40, 200), Y=_log_int(rng, 40, 200), rig=rig)
        del c["name"]
        return c
    bf16 = kind != "backward" and rng.random() < 0.5
    while True:
        Hf, Wf = _log_int(rng, 15, 64), _log_int(rng, 40, 176)
        stride = rng.choice((4, 8))
        if rng.random() < 0.15 and kind == "forward":
            C = rng.randrange(33, 131)  # any channel count
        else:
            C = 8 * rng.choice((4, 6, 8, 10, 12, 16, 16, 20, 24, 32))
        B = rng.choice((1, 1, 1, 2))
        X, Y = _log_int(rng, 48, 512), _log_int(rng, 48, 512)
        Z = _log_int(rng, 4, 64)
        xy = rng.choice((25.0, 50.0, 50.0, 51.2, 100.0))
        if kind == "backward" or kind == "pyramid":
            Z = min(Z, 16)
        if B * X * Y * Z * C <= _MOST_SAMPLES and B * X * Y * C <= (_MOST_OUT if kind == "forward" else _MOST_OUT // 4):
            break
    c = _vt("", kind, B=B, N=rng.choice((4, 5, 6, 6, 6, 7, 8)), C=C, dtype="bf16" if bf16 else "f32", Hf=Hf, Wf=Wf, Himg=Hf * stride,
            Wimg=Wf * stride, X=X, Y=Y, Z=Z, xy=xy, reduce=rng.choice((SUM, MEAN, EQ1)), rig=rig)
    if kind == "forward":
        c["layout"] = rng.choice(("nhwc", "nhwc", "nhwc", "nhwc", "nchw"))
        c["out"] = "bf16" if bf16 and rng.random() < 0.3 else "f32"
        c["count"] = rng.random() < 0.2
    if kind == "pyramid":
        c["levels"] = rng.choice((2, 3, 4))
    del c["name"]
    return c


def _matrices(case, seed):
    rng = np.random.default_rng([int(seed), 1])
    B, N, img = case["B"], case["N"], (case["Himg"], case["Wimg"])
    if case["rig"] == "calibrated":
        m = wl.general_rig(B, N, img, rng, case.get("fov", 70.0))
    else:
        m = wl.ring_rig(N, case.get("fov", 70.0), img, np.deg2rad(rng.uniform(-2.0, 2.0, (B, N))))
    return torch.from_numpy(m).cuda()


def _levels(case):
    """(height, width) of every map of a pyramid."""
    hw = [(case["Hf"], case["Wf"])]
    while len(hw) < case["levels"]:
        hw.append(((hw[-1][0] + 1) // 2, (hw[-1][1] + 1) // 2))
    return hw


def _sca_levels(case):
    h, w = case["Himg"] // case["stride"], case["Wimg"] // case["stride"]
    return [(-(-h // 2 ** i), -(-w // 2 ** i)) for i in range(case["L"])]


def prepare(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7 + 3)

    def normal(*shape):
        return torch.randn(*shape, generator=g, device="cuda", dtype=torch.float32)

    s = dict(kind=case["kind"], lidar2img=_matrices(case, seed), img_hw=(case["Himg"], case["Wimg"]),
             bev_range=(-case["xy"], case["xy"], -case["xy"], case["xy"], case["z0"], case["z1"]))
    B, N, X, Y = case["B"], case["N"], case["X"], case["Y"]
    dt = torch.bfloat16 if case["dtype"] == "bf16" else torch.float32
    if case["kind"] == "sca":
        heads, L, P = case["heads"], case["L"], case["P"]
        lv = _sca_levels(case)
        s["grid"], s["level_hw"] = (X, Y, case["Zref"]), lv
        s["value"] = normal(B, N, sum(h * w for h, w in lv), heads, case["Dh"]).to(dt)
        s["offsets"] = normal(B, X * Y, heads, L, P, 2) * 2.0
        s["weights"] = torch.softmax(normal(B, X * Y, heads, L * P), -1).reshape(B, X * Y, heads, L, P).contiguous()
        return s
    s["grid"], s["reduce"] = (X, Y, case["Z"]), case["reduce"]
    if case["kind"] == "backward":
        s["feat_hw"] = (case["Hf"], case["Wf"])
        s["grad_out"] = normal(B, X, Y, case["C"])
        return s
    planar = case["layout"] == "nchw"
    maps = [normal(*((B, N, case["C"], h, w) if planar else (B, N, h, w, case["C"]))).to(dt) for h, w in _levels(case)]
    if case["kind"] == "pyramid":
        s["features"] = maps
        return s
    s["features"] = maps[0]
    s["layout"] = fb.NCHW if planar else fb.NHWC
    s["out_dtype"] = fb.BF16 if case["out"] == "bf16" else fb.F32
    s["count"] = torch.empty(B, X, Y, dtype=torch.int32, device="cuda") if case["count"] else None
    return s


def run(state):
    s = state
    if s["kind"] == "forward":
        out = fb.sampling_vt(s["features"], s["lidar2img"], s["img_hw"], s["bev_range"], s["grid"], reduce=s["reduce"],
                             valid_count=s["count"], layout=s["layout"], out_dtype=s["out_dtype"])
        return out if s["count"] is None else (out, s["count"])
    if s["kind"] == "backward":
        return fb.sampling_vt_backward(s["grad_out"], s["lidar2img"], s["feat_hw"], s["img_hw"], s["bev_range"], s["grid"], s["reduce"])
    if s["kind"] == "pyramid":
        return fb.sampling_vt_multires(s["features"], s["lidar2img"], s["img_hw"], s["bev_range"], s["grid"], reduce=s["reduce"])
    return fb.sca(s["value"], s["level_hw"], s["lidar2img"], s["offsets"], s["weights"], s["img_hw"], s["bev_range"], s["grid"])


def work(case):
    """Bytes: every input read once and every output written once.  Flops: a surround rig sees a point of the grid in
    about one camera, so about one bilinear sample (four taps) per cell and height bin."""
    e = 2 if case["dtype"] == "bf16" else 4
    B, N, X, Y = case["B"], case["N"], case["X"], case["Y"]
    if case["kind"] == "sca":
        D, pts = case["heads"] * case["Dh"], case["heads"] * case["L"] * case["P"]
        value = B * N * sum(h * w for h, w in _sca_levels(case)) * D * e
        return {"bytes": value + B * N * 64 + B * X * Y * (pts * 12 + D * 4), "flops": B * X * Y * pts * case["Dh"] * 8}
    C = case["C"]
    maps = sum(B * N * h * w * C * e for h, w in _levels(case))
    out = B * X * Y * (C * (2 if case["out"] == "bf16" else 4) + (4 if case["count"] else 0))
    return {"bytes": maps + B * N * 64 + out, "flops": B * X * Y * case["Z"] * C * 8 * case["levels"]}


def tolerance(case):
    """Sums in single precision, in any order; results asked for in bf16 may round to the neighbouring value."""
    if case.get("out") == "bf16":
        return {"rel": 3e-3, "max": 1e-2}
    return {"rel": 1e-5}
