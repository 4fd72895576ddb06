"""Kernels that start before the one before them has ended -- of one call (planar and ragged tensors after the copy of their
features, pyramid levels after the level before) and of calls that follow one another: inputs that the stream has only just
written, and buffers that it uses again, give what the same calls give on an idle GPU."""
import numpy as np
import pytest

from paper_2607_10071_b200 import binding as fb
from paper_2607_10071_b200 import workloads as wl

pytestmark = pytest.mark.gpu

W = wl.Workload("early", 9300, 1, 6, 48, "f32", (20, 36), (160, 288), (70, 66, 8), (-25.0, 25.0, -25.0, 25.0, -4.0, 3.0), 0, general_pose=True)


def calls(kind, feats, mats, work):
    args = (mats, W.img_hw, W.bev_range, W.grid)
    if kind == "planar":
        return fb.sampling_vt(feats[0], *args, layout=fb.NCHW, workspace=work)
    if kind == "ragged":
        return fb.sampling_vt(feats[0], *args, reduce=2, workspace=work)
    if kind == "planar pyramid":
        return fb.sampling_vt_multires(feats, *args, reduce=1, layout=fb.NCHW)
    return fb.sampling_vt_multires(feats, *args, reduce=2)


@pytest.mark.parametrize("kind", ["planar", "ragged", "pyramid", "planar pyramid"])
def test_inputs_written_just_before_the_call(kind):
    import torch
    dev = torch.device("cuda:0")
    C, (h, w) = (46 if kind == "ragged" else 48), W.feat_hw
    levels = [(h, w), (h // 2, w // 2), (h // 4, w // 4)] if "pyramid" in kind else [(h, w)]
    shapes = [(1, 6, C, a, b) if "planar" in kind else (1, 6, a, b, C) for a, b in levels]
    g = torch.Generator(device=dev).manual_seed(7)
    rounds = 12
    src = [[torch.randn(s, generator=g, device=dev) for s in shapes] for _ in range(rounds)]
    rigs = [torch.from_numpy(wl.general_rig(1, 6, W.img_hw, np.random.default_rng(i))).to(dev) for i in range(rounds)]
    work = torch.empty(64 << 20, dtype=torch.uint8, device=dev)
    want = []
    for f, m in zip(src, rigs):
        want.append(calls(kind, f, m, work).clone())
        torch.cuda.synchronize()
    feats, mats = [torch.empty(s, device=dev) for s in shapes], torch.empty_like(rigs[0])
    big = torch.randn(2048, 2048, device=dev)
    got = []
    for i in range(rounds):
        if i % 3 == 0:
            big = (big @ big) * 1e-3  # (the queue fills up: the kernels of the calls stand behind one another)
        for t, s in zip(feats, src[i]):
            t.copy_(s)
        mats.copy_(rigs[i])
        got.append(calls(kind, feats, mats, work))
    torch.cuda.synchronize()
    for i in range(rounds):
        assert torch.equal(got[i], want[i]), (kind, i, float((got[i] - want[i]).abs().max()))


# ---- one call feeds the next, with nothing between them
ROUNDS = 6


class Chain:
    """``ROUNDS`` rounds of calls.  A round has inputs of its own and hands every result on to the call after it, through buffers
    that all rounds share; what a round is judged by (``results``) goes to tensors of its own."""

    def __init__(self, blocks):
        import torch
        self.dev = torch.device("cuda:0")
        self.gen = torch.Generator(device=self.dev).manual_seed(11)
        self.tune = (0, 0, 16, 0) if blocks == "scatter" else (0, 0, 0, 0)
        # 216 texel columns over 4620 cells: a CTA each; 36 over 21000: five share one, and a memset comes before them
        self.N, self.grid = (1, (150, 140, 8)) if blocks == "several" else (6, (70, 66, 8))
        self.feat, self.img, self.range = (20, 36), (160, 288), W.bev_range
        self.rigs = [torch.from_numpy(wl.general_rig(1, self.N, self.img, np.random.default_rng(i))).to(self.dev) for i in range(ROUNDS)]
        self.names = []

    def normal(self, *shape):
        import torch
        return torch.randn(*shape, generator=self.gen, device=self.dev)

    def empty(self, *shape):
        import torch
        return torch.full(shape, float("nan"), device=self.dev)

    def per_round(self, *shape):
        return [self.empty(*shape) for _ in range(ROUNDS)]

    def forward(self, i, features, out, **k):
        fb.sampling_vt(features, self.rigs[i], self.img, self.range, self.grid, 2, out=out, **k)

    def backward(self, i, grad_out, grad):
        fb.sampling_vt_backward(grad_out, self.rigs[i], self.feat, self.img, self.range, self.grid, 2, grad_features=grad, tune=self.tune)
        self.names.append(fb.flashbev_last_kernel_name())


class ForwardBackward(Chain):
    """An output is the next grad_out, a gradient the next features."""

    def __init__(self, blocks):
        super().__init__(blocks)
        maps, cells, C = (1, self.N) + self.feat, (1,) + self.grid[:2], 48
        self.features, self.grad, self.again = [self.normal(*maps, C) for _ in range(ROUNDS)], self.empty(*maps, C), self.empty(*cells, C)
        self.first, self.second, self.last = self.per_round(*cells, C), self.per_round(*cells, C), self.per_round(*maps, C)
        self.results = [self.first, self.second, self.last]

    def round(self, i):
        self.forward(i, self.features[i], self.first[i])
        self.backward(i, self.first[i], self.grad)
        self.forward(i, self.grad, self.second[i])
        self.forward(i, self.grad, self.again)
        self.backward(i, self.again, self.grad)      # (what the call before reads)
        self.backward(i, self.second[i], self.last[i])


class Attention(Chain):
    """The cross-attention's output is a grad_out, the gradient the next cross-attention's values."""

    def __init__(self, blocks):
        super().__init__(blocks)
        X, Y, _ = self.grid
        heads, Dh, P, (h, w) = 8, 32, 4, self.feat
        self.value = [self.normal(1, self.N, h * w, heads, Dh) for _ in range(ROUNDS)]
        self.offsets = self.normal(1, X * Y, heads, 1, P, 2) * 2.0
        self.weights = self.normal(1, X * Y, heads, 1, P).softmax(-1)
        self.out, self.grad = self.empty(1, X * Y, heads * Dh), self.empty(1, self.N, h, w, heads * Dh)
        self.first, self.last = self.per_round(1, self.N, h, w, heads * Dh), self.per_round(1, X * Y, heads * Dh)
        self.results = [self.first, self.last]

    def attend(self, i, value, out):
        fb.sca(value, [self.feat], self.rigs[i], self.offsets, self.weights, self.img, self.range, self.grid[:2] + (4,), out=out)

    def round(self, i):
        cells = self.out.view(1, *self.grid[:2], -1)
        self.attend(i, self.value[i], self.out)
        self.backward(i, cells, self.first[i])
        self.attend(i, self.first[i].view(self.value[i].shape), self.out)
        self.backward(i, cells, self.grad)
        self.attend(i, self.grad.view(self.value[i].shape), self.last[i])


class Pyramid(Chain):
    """A pyramid's output is a grad_out, the gradient the finest level of the next pyramid."""

    def __init__(self, blocks):
        super().__init__(blocks)
        (h, w), C = self.feat, 48
        self.levels = [[self.normal(1, self.N, h >> s, w >> s, C) for s in range(3)] for _ in range(ROUNDS)]
        self.grad, self.first, self.last = self.empty(1, self.N, h, w, C), self.empty(1, *self.grid[:2], C), self.per_round(1, *self.grid[:2], C)
        self.results = [self.last]

    def sum(self, i, levels, out):
        fb.sampling_vt_multires(levels, self.rigs[i], self.img, self.range, self.grid, reduce=2, out=out)

    def round(self, i):
        self.sum(i, self.levels[i], self.first)
        self.backward(i, self.first, self.grad)
        self.sum(i, [self.grad] + self.levels[i][1:], self.last[i])


class LentWorkspace(Chain):
    """Planar and ragged calls in a row with one workspace; a planar output is the next planar call's input where it fits."""

    def __init__(self, blocks):
        super().__init__(blocks)
        import torch
        h, w = self.feat
        self.planar = [self.normal(1, self.N, 48, h, w) for _ in range(ROUNDS)]
        self.ragged = [self.normal(1, self.N, h, w, 46) for _ in range(ROUNDS)]
        self.work = torch.empty(4 << 20, dtype=torch.uint8, device=self.dev)
        cells = self.grid[:2]
        self.first, self.second, self.last = self.per_round(1, 48, *cells), self.per_round(1, *cells, 46), self.per_round(1, 48, *cells)
        self.results = [self.first, self.second, self.last]

    def round(self, i):
        self.forward(i, self.planar[i], self.first[i], layout=fb.NCHW, workspace=self.work)
        self.names.append(fb.flashbev_last_kernel_name())
        self.forward(i, self.ragged[i], self.second[i], workspace=self.work)
        self.names.append(fb.flashbev_last_kernel_name())
        features = self.first[i].view(-1)[:self.planar[i].numel()].view(self.planar[i].shape)
        self.forward(i, features, self.last[i], layout=fb.NCHW, workspace=self.work)


@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("kind,blocks", [(k, b) for k in (ForwardBackward, Attention, Pyramid) for b in ("one", "several", "scatter")] +
                         [(LentWorkspace, "one"), (LentWorkspace, "several")])
def test_calls_that_feed_one_another(kind, blocks, graph):
    """In a stream behind other work, and in a graph.  The order of the backward's sums changes from run to run: each run is
    within 2e-6 of the exact gradient (relative 2-norm; `test_gpu_backward`), and what the later calls make of the difference
    keeps its size, since they are linear in it: 4e-6 for each of at most two backward calls, with as much again of room.  A value
    that was not waited for is another round's or NaN: an error of the order of the value itself, which the largest difference of
    one element finds."""
    import torch
    chain = kind(blocks)
    chain.round(0)
    torch.cuda.synchronize()
    if kind is LentWorkspace:
        assert chain.names == ["tiled_f32_nchw", "tiled_f32_padded"]
    else:
        assert all(("texel" in name) == (blocks != "scatter") for name in chain.names), chain.names
    want = []
    for i in range(ROUNDS):
        chain.round(i)
        torch.cuda.synchronize()
        want.append([r[i].clone() for r in chain.results])
    for r in chain.results:
        for t in r:
            t.fill_(float("nan"))
    if graph:
        stream, g = torch.cuda.Stream(), torch.cuda.CUDAGraph()
        stream.wait_stream(torch.cuda.current_stream())
        with torch.cuda.graph(g, stream=stream):
            for i in range(ROUNDS):
                chain.round(i)
        for _ in range(3):
            g.replay()
    else:
        big = torch.randn(4096, 4096, device=chain.dev)
        for _ in range(3):
            big = (big @ big) * 1e-3  # (the queue fills up: the kernels stand behind one another)
        for i in range(ROUNDS):
            chain.round(i)
    torch.cuda.synchronize()
    for i in range(ROUNDS):
        for at, r in enumerate(chain.results):
            got, ref = r[i].double(), want[i][at].double()
            if kind is LentWorkspace or (kind is ForwardBackward and at == 0):  # (no sum in an order that changes)
                assert torch.equal(got, ref), (kind, i, at)
            err = got - ref
            assert float(err.norm()) <= 4 * 4e-6 * float(ref.norm()), (kind, i, at, float(err.norm() / ref.norm()))
            assert float(err.abs().max()) <= 1e-3 * float(ref.abs().max()), (kind, i, at)
