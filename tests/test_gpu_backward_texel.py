"""The texel-side backward kernel at the sizes where it can go wrong: edges of its row tiles (16 and 64 rows), channel tiles
(80 channels, 8 per fragment) and channel blocks, maps of one texel, one and two CTAs per texel column, and gradients that are
not finite.  Tolerances are those of the backward's other tests (`test_gpu_backward`), the same bounds for both kernels."""
import numpy as np
import pytest

from paper_2607_10071_b200 import binding as fb
from paper_2607_10071_b200 import build as fbuild
from paper_2607_10071_b200 import workloads as wl
from tests.test_gpu_backward import check, run_backward

pytestmark = pytest.mark.gpu
SUM, MEAN, EQ1 = 0, 1, 2
SCATTER = (0, 0, 16, 0)  # hints select the scatter kernel


def workload(name, C, feat, grid, general=True, B=1, N=6, xy=25.0, reduce=0):
    return wl.Workload(name, 9100 + C, B, N, C, "f32", feat, (feat[0] * 8, feat[1] * 8), grid, (-xy, xy, -xy, xy, -4.0, 3.0), reduce,
                       general_pose=general)


@pytest.mark.parametrize("feat", [(1, 1), (1, 9), (15, 7), (16, 12), (17, 30), (32, 20), (33, 11), (64, 10), (65, 10), (130, 6)])
@pytest.mark.parametrize("reduce", [SUM, MEAN, EQ1])
def test_row_tiles(oracle, feat, reduce):
    for general in (False, True):
        w = workload("rows", 44, feat, (37, 41, 9), general)
        assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce, seed=feat[0])


@pytest.mark.parametrize("C", [4, 8, 12, 16, 32, 36, 80, 84, 96, 128, 132, 160, 164, 320, 324, 644])
def test_channel_tiles(oracle, C):
    w = workload("channels", C, (18, 26), (29, 33, 6), B=2, N=3)
    reduce = C // 4 % 3 if C > 40 else SUM  # (few channels in the mean modes: the scatter)
    assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce, seed=C)


@pytest.mark.parametrize("C", [4, 32, 36, 48, 64, 80, 100, 128, 132])
@pytest.mark.parametrize("rows", [33, 48, 49, 64])
def test_two_row_tiles_per_warp(oracle, C, rows):
    """Three and four row tiles: up to 128 channels a warp has two of them, unless that pads the channels much further (36, 48)."""
    w = workload("two_tiles", C, (rows, 14), (23, 27, 12), general=C % 8 == 0, N=4)
    assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, SUM, seed=rows)


@pytest.mark.parametrize("Z", [1, 2, 3, 5, 63, 64])
def test_height_bins(oracle, Z):
    w = workload("bins", 48, (20, 24), (31, 30, Z), N=5)
    for reduce in (SUM, MEAN, EQ1):
        assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce, seed=Z)


@pytest.mark.parametrize("general", [False, True])
def test_two_blocks_per_column_and_a_full_list(oracle, general):
    """Few texel columns over many cells: two CTAs share a column, and its cells do not fit the list at once."""
    w = workload("long_lists", 48, (24, 10), (220, 190, 4), general, N=2, xy=40.0)
    for reduce in (SUM, EQ1):
        assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce)


@pytest.mark.parametrize("N,feat,grid", [(1, (7, 1), (60, 50, 3)), (1, (32, 9), (97, 64, 5)), (1, (64, 28), (90, 101, 4)),
                                         (2, (33, 31), (181, 130, 4)), (3, (20, 25), (61, 47, 6))])
def test_several_blocks_per_column(oracle, N, feat, grid):
    """As few columns as leave SMs without one: up to eight CTAs share a column, some of them with no cell at all."""
    for C, reduce in ((48, SUM), (132, EQ1), (160, MEAN)):
        w = workload("shared", C, feat, grid, N=N, xy=30.0)
        assert "texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce)


@pytest.mark.parametrize("C,feat,grid,reduce", [(128, (32, 28), (227, 222, 8), EQ1), (128, (64, 21), (443, 118, 4), EQ1),
                                                (80, (32, 40), (512, 512, 8), SUM)])
def test_few_columns_are_not_left_to_few_blocks(C, feat, grid, reduce):
    """One camera over a large grid: the scatter has work for every SM, so the texel side must not be slower than it (with two
    CTAs per column it took 1.2 to 1.6 times as long; measured 0.5 to 0.6 now, asserted with room for other clocks)."""
    import torch
    w = workload("few", C, feat, grid, N=1, xy=50.0)
    dev = torch.device("cuda:0")
    m = torch.from_numpy(wl.make_inputs(w).lidar2img).to(dev)
    g = torch.randn((1,) + tuple(grid[:2]) + (C,), device=dev)
    out = torch.empty((1, 1) + feat + (C,), device=dev)

    def time(tune):
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                fb.sampling_vt_backward(g, m, feat, w.img_hw, w.bev_range, grid, reduce, grad_features=out, tune=tune)
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) / 20)
        return best, fb.flashbev_last_kernel_name()

    (texel, name), (scatter, other) = time((0, 0, 0, 0)), time((0, 0, 16, 0))
    assert "texel" in name and "texel" not in other
    assert texel <= 1.1 * scatter, (texel, scatter)


@pytest.mark.parametrize("C,N,B,feat,grid,texel", [(80, 8, 2, (63, 84), (28, 47, 2), False), (64, 7, 1, (55, 144), (75, 53, 4), False),
                                                   (128, 6, 1, (10, 167), (86, 47, 2), False), (44, 5, 1, (20, 160), (60, 80, 5), True),
                                                   (44, 5, 1, (20, 160), (60, 79, 5), False), (48, 5, 1, (20, 24), (31, 30, 1), True),
                                                   (44, 1, 66000, (1, 1), (1, 1, 1), True)])
def test_many_columns_with_little_for_each(oracle, C, N, B, feat, grid, texel):
    """More columns than the SMs hold at once take 30 samples each or go to the scatter, which had been up to 2.9 times as fast; what
    the scatter refuses (65536 batch elements) stays accepted."""
    for reduce in (SUM, MEAN, EQ1):
        w = workload("little", C, feat, grid, N=N, B=B)
        assert ("texel" in check(oracle, w, wl.make_inputs(w).lidar2img, reduce)) == texel


def test_many_cameras_see_every_cell(oracle):
    w = workload("cameras", 44, (16, 20), (24, 22, 7), N=33)
    inp = wl.make_inputs(w)
    inp.lidar2img[:] = inp.lidar2img[:, :1]
    for reduce in (SUM, MEAN, EQ1):
        assert "texel" in check(oracle, w, inp.lidar2img, reduce)


@pytest.mark.parametrize("C,feat,reduce", [(16, (20, 26), SUM), (32, (16, 22), SUM), (48, (18, 30), MEAN), (64, (32, 44), EQ1),
                                           (80, (32, 44), SUM), (132, (30, 25), EQ1), (64, (47, 21), SUM), (128, (56, 50), EQ1)])
def test_a_single_product_is_rounded_once(C, feat, reduce):
    """Channels that one cell alone has a gradient in: two per cell, 1 in the one -- the result is the texel's weight, as it
    stands in single precision -- and any number in the other, whose result is then one product.  It is rounded once (2^-24 of
    it, half an ulp) and lacks the smallest products of its pieces (2^-24 at most); what the tensor cores cut off the others
    is below 2^-27.  Root mean square: 2.53e-8 for the rounding (2^-24 / sqrt(3), over significands of 1 to 2), 0.6e-8 for the
    rest, 2.6e-8 together; a thousand values are within a tenth of it."""
    w = workload("single", C, feat, (40, 37, 5), reduce=reduce)
    m = wl.make_inputs(w).lidar2img
    rng = np.random.default_rng(C)
    off = []
    for _ in range(8):
        G = np.zeros((1,) + tuple(w.grid[:2]) + (C,), np.float32)
        g = (rng.uniform(1.0, 2.0, C // 2) * 2.0 ** rng.integers(-20, 20, C // 2) * rng.choice((-1, 1), C // 2)).astype(np.float32)
        for c in range(C // 2):
            x, y = rng.integers(w.grid[0]), rng.integers(w.grid[1])
            G[0, x, y, 2 * c], G[0, x, y, 2 * c + 1] = 1.0, g[c]
        got, name = run_backward(w, m, G, reduce)
        assert "texel" in name
        weight, result = got[..., 0::2].astype(np.float64), got[..., 1::2].astype(np.float64)
        exact = weight * g.astype(np.float64)
        assert np.array_equal(weight != 0.0, result != 0.0)
        off.append(np.abs(result - exact)[weight != 0.0] / np.abs(exact[weight != 0.0]))
    off = np.concatenate(off)
    assert off.size > 1000
    assert off.max() <= 2.0 ** -23 + 2.0 ** -27 and np.sqrt((off ** 2).mean()) <= 2.9e-8, (off.max(), np.sqrt((off ** 2).mean()))


@pytest.mark.parametrize("shared", [False, True])
def test_gradients_that_are_not_finite(shared):
    """Infinite and NaN output gradients reach the texels that their cell weighs and no others, as in the scatter."""
    w = workload("nonfinite", 44, (24, 10), (220, 190, 4), N=2) if shared else workload("nonfinite", 84, (33, 20), (40, 40, 6))
    m = wl.make_inputs(w).lidar2img
    rng = np.random.default_rng(5)
    G = rng.standard_normal((w.B,) + tuple(w.grid[:2]) + (w.C,)).astype(np.float32)
    for value, cells in ((np.inf, 3), (-np.inf, 3), (np.nan, 2), (3.4e38, 2)):
        for _ in range(cells):
            G[0, rng.integers(w.grid[0]), rng.integers(w.grid[1]), rng.integers(w.C)] = value
    for reduce in (SUM, MEAN, EQ1):
        got, name = run_backward(w, m, G, reduce)
        ref, other = run_backward(w, m, G, reduce, SCATTER)
        assert "texel" in name and "texel" not in other
        assert np.array_equal(np.isnan(got), np.isnan(ref)) and np.array_equal(np.isposinf(got), np.isposinf(ref))
        assert np.array_equal(np.isneginf(got), np.isneginf(ref)) and not np.isfinite(ref).all()
        ok = np.isfinite(ref)
        # two fp32 sums of the same numbers: 2e-6 of the result each (test_gpu_backward), per channel (the large value stands alone)
        err = np.where(ok, got, 0.0).astype(np.float64) - np.where(ok, ref, 0.0)
        assert np.all(np.sqrt((err ** 2).sum((0, 1, 2, 3))) <= 4e-6 * np.sqrt((np.where(ok, ref, 0.0).astype(np.float64) ** 2).sum((0, 1, 2, 3))))


@pytest.mark.parametrize("reduce", [SUM, MEAN, EQ1])
def test_makes_no_out_of_range_index(reduce):
    import torch
    lib = fb.load_library(fbuild.build(debug_bounds=True))
    dev = torch.device("cuda:0")
    for C, feat, grid, N in ((44, (65, 10), (37, 41, 9), 6), (132, (17, 30), (64, 48, 5), 4), (48, (24, 10), (220, 190, 4), 2)):
        w = workload("bounds", C, feat, grid, N=N)
        m = torch.from_numpy(wl.make_inputs(w).lidar2img).to(dev)
        g = torch.randn((1,) + tuple(grid[:2]) + (C,), device=dev)
        g[0, 3, 3, 1] = float("inf")
        out, err = torch.empty((1, N) + feat + (C,), device=dev), torch.zeros(1, dtype=torch.int32, device=dev)
        p = fb.make_backward_params(g.data_ptr(), m.data_ptr(), 1, N, C, feat, w.img_hw, w.bev_range, grid, reduce, out.data_ptr(),
                                    debug_error_word=err.data_ptr())
        fb.flashbev_sampling_vt_backward(p, torch.cuda.current_stream().cuda_stream, library=lib)
        assert err.item() == 0 and lib.flashbev_last_kernel_name() == b"tiled_bwd_texel"
