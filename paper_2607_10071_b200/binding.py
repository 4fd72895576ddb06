"""Thin binding of the C ABI in include/flashbev.h.

Argument marshalling only: every step of the operator runs inside the CUDA
library.  PyTorch is used by callers for device memory and streams; the ctypes
part of this module needs only integer addresses, the functions for torch
tensors (``sampling_vt`` and the like) marshal in the extension module
``_native`` (csrc/native.cpp).  There is no CPU fallback: if the library has not
been built, or the call fails, an exception is raised.
"""
from __future__ import annotations

import ctypes
import os

_HERE = os.path.dirname(os.path.abspath(__file__))
LIB_PATH = os.path.join(_HERE, "libflashbev.so")

OK, INVALID_ARG, UNSUPPORTED, MISALIGNED, CUDA_ERROR, TOO_SMALL = range(6)
EXCEEDS_STATIC_STAGING = 6
STATIC_STAGING_BYTES = 32 * 1024 * 1024
F32, BF16 = 0, 1
NHWC, NCHW = 0, 1
REDUCE_SUM, REDUCE_MEAN_OVER_VALID, REDUCE_CAMERA_MEAN_Z_SUM = 0, 1, 2
KERNEL_AUTO, KERNEL_PER_OUTPUT, KERNEL_TILED = 0, 1, 2


class VtParams(ctypes.Structure):
    """Mirror of ``flashbev_vt_params``."""
    _fields_ = [
        ("struct_size", ctypes.c_size_t),
        ("features", ctypes.c_void_p),
        ("feat_dtype", ctypes.c_int32),
        ("layout", ctypes.c_int32),
        ("lidar2img", ctypes.c_void_p),
        ("B", ctypes.c_int32), ("N", ctypes.c_int32), ("C", ctypes.c_int32),
        ("feat_h", ctypes.c_int32), ("feat_w", ctypes.c_int32),
        ("img_h", ctypes.c_int32), ("img_w", ctypes.c_int32),
        ("x_min", ctypes.c_double), ("x_max", ctypes.c_double),
        ("y_min", ctypes.c_double), ("y_max", ctypes.c_double),
        ("z_min", ctypes.c_double), ("z_max", ctypes.c_double),
        ("X", ctypes.c_int32), ("Y", ctypes.c_int32), ("Z", ctypes.c_int32),
        ("reduce", ctypes.c_int32),
        ("out", ctypes.c_void_p),
        ("out_dtype", ctypes.c_int32),
        ("kernel", ctypes.c_int32),
        ("valid_count_out", ctypes.c_void_p),
        ("tune", ctypes.c_int32 * 4),
        ("debug_error_word", ctypes.c_void_p),
        ("workspace", ctypes.c_void_p),
        ("workspace_bytes", ctypes.c_size_t),
    ]


class VtBackwardParams(ctypes.Structure):
    """Mirror of ``flashbev_vt_backward_params``."""
    _fields_ = [
        ("struct_size", ctypes.c_size_t),
        ("grad_out", ctypes.c_void_p),
        ("lidar2img", ctypes.c_void_p),
        ("B", ctypes.c_int32), ("N", ctypes.c_int32), ("C", ctypes.c_int32),
        ("feat_h", ctypes.c_int32), ("feat_w", ctypes.c_int32),
        ("img_h", ctypes.c_int32), ("img_w", ctypes.c_int32),
        ("x_min", ctypes.c_double), ("x_max", ctypes.c_double),
        ("y_min", ctypes.c_double), ("y_max", ctypes.c_double),
        ("z_min", ctypes.c_double), ("z_max", ctypes.c_double),
        ("X", ctypes.c_int32), ("Y", ctypes.c_int32), ("Z", ctypes.c_int32),
        ("reduce", ctypes.c_int32),
        ("grad_features", ctypes.c_void_p),
        ("tune", ctypes.c_int32 * 4),
        ("debug_error_word", ctypes.c_void_p),
    ]


class ScaParams(ctypes.Structure):
    """Mirror of ``flashbev_sca_params``."""
    _fields_ = [
        ("struct_size", ctypes.c_size_t),
        ("value", ctypes.c_void_p),
        ("value_dtype", ctypes.c_int32), ("chunk_records", ctypes.c_int32),
        ("level_hw", ctypes.c_void_p),
        ("lidar2img", ctypes.c_void_p),
        ("offsets", ctypes.c_void_p),
        ("weights", ctypes.c_void_p),
        ("B", ctypes.c_int32), ("N", ctypes.c_int32), ("heads", ctypes.c_int32), ("head_dim", ctypes.c_int32),
        ("L", ctypes.c_int32), ("P", ctypes.c_int32),
        ("img_h", ctypes.c_int32), ("img_w", ctypes.c_int32),
        ("x_min", ctypes.c_double), ("x_max", ctypes.c_double),
        ("y_min", ctypes.c_double), ("y_max", ctypes.c_double),
        ("z_min", ctypes.c_double), ("z_max", ctypes.c_double),
        ("X", ctypes.c_int32), ("Y", ctypes.c_int32), ("Zref", ctypes.c_int32), ("reserved2", ctypes.c_int32),
        ("out", ctypes.c_void_p),
        ("hits_out", ctypes.c_void_p),
    ]


class VtMultiresParams(ctypes.Structure):
    """ctypes mirror of ``flashbev_vt_multires_params``."""
    _fields_ = [
        ("struct_size", ctypes.c_size_t),
        ("base", ctypes.POINTER(VtParams)),
        ("levels", ctypes.c_int32), ("reserved", ctypes.c_int32),
        ("features", ctypes.POINTER(ctypes.c_void_p)),
        ("feat_hw", ctypes.POINTER(ctypes.c_int32)),
    ]


MAX_LEVELS = 8


class FlashBevError(RuntimeError):
    def __init__(self, status: int, what: str):
        super().__init__(f"{what}: {status_string(status)} (status {status})")
        self.status = status


_lib = None


def _declare(L: ctypes.CDLL) -> ctypes.CDLL:
    """Argument and result types of every entry point of a loaded libflashbev."""
    P = ctypes.POINTER(VtParams)
    L.flashbev_sampling_vt.restype = ctypes.c_int
    L.flashbev_sampling_vt.argtypes = [P, ctypes.c_void_p]
    L.flashbev_sampling_vt_host.restype = ctypes.c_int
    L.flashbev_sampling_vt_host.argtypes = [P, ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p]
    L.flashbev_sampling_vt_host_static.restype = ctypes.c_int
    L.flashbev_sampling_vt_host_static.argtypes = [P, ctypes.c_void_p]
    L.flashbev_sampling_vt_backward.restype = ctypes.c_int
    L.flashbev_sampling_vt_backward.argtypes = [ctypes.POINTER(VtBackwardParams), ctypes.c_void_p]
    L.flashbev_sampling_vt_multires.restype = ctypes.c_int
    L.flashbev_sampling_vt_multires.argtypes = [ctypes.POINTER(VtMultiresParams), ctypes.c_void_p]
    L.flashbev_sca.restype = ctypes.c_int
    L.flashbev_sca.argtypes = [ctypes.POINTER(ScaParams), ctypes.c_void_p]
    L.flashbev_workspace_bytes.restype = ctypes.c_size_t
    L.flashbev_workspace_bytes.argtypes = [P]
    L.flashbev_host_staging_bytes.restype = ctypes.c_size_t
    L.flashbev_host_staging_bytes.argtypes = [P]
    L.flashbev_last_launch_count.restype = ctypes.c_int
    L.flashbev_last_kernel_name.restype = ctypes.c_char_p
    L.flashbev_status_string.restype = ctypes.c_char_p
    L.flashbev_status_string.argtypes = [ctypes.c_int]
    L.flashbev_version.restype = ctypes.c_int
    return L


def load_library(path: str) -> ctypes.CDLL:
    """Load another build of the library (e.g. the bounds-checked one) next to the default one."""
    if not os.path.exists(path):
        raise FileNotFoundError(f"{path} is missing: build it with paper_2607_10071_b200.build (there is no CPU fallback)")
    return _declare(ctypes.CDLL(path))


def lib() -> ctypes.CDLL:
    """Load libflashbev.so (built in-tree by ``paper_2607_10071_b200.build``)."""
    global _lib
    if _lib is None:
        if not os.path.exists(LIB_PATH):
            raise FileNotFoundError(
                f"{LIB_PATH} is missing: build it with `python -m paper_2607_10071_b200.build` "
                "(there is no CPU fallback)")
        _lib = _declare(ctypes.CDLL(LIB_PATH))
    return _lib


_native = None


def native():
    """The extension module over libflashbev.so (built in-tree by ``paper_2607_10071_b200.build``)."""
    global _native
    if _native is None:
        import torch  # noqa: F401  (its libraries have to be loaded first)
        try:
            from . import _native as module
        except ImportError as e:
            raise ImportError("the extension module is missing: build it with `python -m paper_2607_10071_b200.build` "
                              "(there is no CPU fallback)") from e
        _native = module
    return _native


def _result(r, what):
    """A result tensor of the extension module, or the status of a refused call raised."""
    if type(r) is int:
        raise FlashBevError(r, what)
    return r


def status_string(status: int) -> str:
    return lib().flashbev_status_string(int(status)).decode()


def version() -> int:
    return int(lib().flashbev_version())


def make_params(features_ptr, feat_dtype, lidar2img_ptr, B, N, C, feat_hw, img_hw, bev_range, grid,
                reduce, out_ptr, valid_count_ptr=None, kernel=KERNEL_AUTO, tune=(0, 0, 0, 0),
                layout=NHWC, out_dtype=F32, debug_error_word=None, workspace=None, workspace_bytes=0) -> VtParams:
    p = VtParams()
    p.struct_size = ctypes.sizeof(VtParams)
    p.features, p.feat_dtype, p.layout = features_ptr, feat_dtype, layout
    p.lidar2img = lidar2img_ptr
    p.B, p.N, p.C = B, N, C
    p.feat_h, p.feat_w = feat_hw
    p.img_h, p.img_w = img_hw
    p.x_min, p.x_max, p.y_min, p.y_max, p.z_min, p.z_max = (float(v) for v in bev_range)
    p.X, p.Y, p.Z = grid
    p.reduce = reduce
    p.out, p.out_dtype, p.kernel = out_ptr, out_dtype, kernel
    p.valid_count_out = valid_count_ptr
    p.debug_error_word = debug_error_word
    p.workspace, p.workspace_bytes = workspace, int(workspace_bytes)
    for i, t in enumerate(tune):
        p.tune[i] = int(t)
    return p


def flashbev_sampling_vt(params: VtParams, stream: int | None = None, check: bool = True, library=None) -> int:
    """Enqueue the fused operator on ``stream`` (a raw cudaStream_t value; None/0 = default stream).
    ``library``: another build loaded with ``load_library`` instead of the default one."""
    st = (library or lib()).flashbev_sampling_vt(ctypes.byref(params), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sampling_vt")
    return st


def flashbev_sampling_vt_host(params: VtParams, d_staging: int, staging_bytes: int, stream: int | None = None,
                              check: bool = True) -> int:
    """Host-buffer variant: pointers in ``params`` are host addresses, ``d_staging`` a device buffer."""
    st = lib().flashbev_sampling_vt_host(ctypes.byref(params), ctypes.c_void_p(d_staging),
                                         ctypes.c_size_t(staging_bytes), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sampling_vt_host")
    return st


def flashbev_sampling_vt_host_static(params: VtParams, stream: int | None = None, check: bool = True) -> int:
    """Host-buffer variant for callers that may not allocate device memory: pointers in ``params`` are
    host addresses and the staging area is the fixed STATIC_STAGING_BYTES array inside the library.
    Calls on one device must not overlap on the GPU (they share that array)."""
    st = lib().flashbev_sampling_vt_host_static(ctypes.byref(params), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sampling_vt_host_static")
    return st


def flashbev_sampling_vt_multires(base: VtParams, feature_ptrs, feat_hws, stream: int | None = None,
                                  check: bool = True) -> int:
    """Sum of the operator over the levels of a feature pyramid: ``feature_ptrs`` are device pointers,
    ``feat_hws`` the (feat_h, feat_w) of every level; ``base`` carries everything else."""
    n = len(feature_ptrs)
    q = VtMultiresParams()
    q.struct_size = ctypes.sizeof(VtMultiresParams)
    q.base = ctypes.pointer(base)
    q.levels = n
    ptrs = (ctypes.c_void_p * max(n, 1))(*[int(v) for v in feature_ptrs])
    hw = (ctypes.c_int32 * max(2 * n, 2))(*[int(v) for pair in feat_hws for v in pair])
    q.features = ctypes.cast(ptrs, ctypes.POINTER(ctypes.c_void_p))
    q.feat_hw = ctypes.cast(hw, ctypes.POINTER(ctypes.c_int32))
    st = lib().flashbev_sampling_vt_multires(ctypes.byref(q), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sampling_vt_multires")
    return st


def make_backward_params(grad_out_ptr, lidar2img_ptr, B, N, C, feat_hw, img_hw, bev_range, grid, reduce,
                         grad_features_ptr, tune=(0, 0, 0, 0), debug_error_word=None) -> VtBackwardParams:
    p = VtBackwardParams()
    p.struct_size = ctypes.sizeof(VtBackwardParams)
    p.grad_out, p.lidar2img, p.grad_features = grad_out_ptr, lidar2img_ptr, grad_features_ptr
    p.B, p.N, p.C = B, N, C
    p.feat_h, p.feat_w = feat_hw
    p.img_h, p.img_w = img_hw
    p.x_min, p.x_max, p.y_min, p.y_max, p.z_min, p.z_max = (float(v) for v in bev_range)
    p.X, p.Y, p.Z = grid
    p.reduce = reduce
    for i, t in enumerate(tune):
        p.tune[i] = int(t)
    p.debug_error_word = debug_error_word
    return p


def flashbev_sampling_vt_backward(params: VtBackwardParams, stream: int | None = None, check: bool = True,
                                  library=None) -> int:
    """Enqueue the gradient w.r.t. the features (one kernel, after a memset where blocks share texels) on ``stream``."""
    st = (library or lib()).flashbev_sampling_vt_backward(ctypes.byref(params), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sampling_vt_backward")
    return st


def sampling_vt_backward(grad_out, lidar2img, feat_hw, img_hw, bev_range, grid, reduce=REDUCE_SUM,
                         grad_features=None, tune=(0, 0, 0, 0), stream=None):
    """grad_out: CUDA float32 [B,X,Y,C]; returns CUDA float32 [B,N,Hf,Wf,C] (marshalling only)."""
    return _result((_native or native()).sampling_vt_backward(grad_out, lidar2img, feat_hw, img_hw, bev_range, grid, reduce,
                                                              grad_features, tune, stream), "flashbev_sampling_vt_backward")


def flashbev_sca(params: ScaParams, stream: int | None = None, check: bool = True) -> int:
    """Enqueue the fused spatial cross-attention on ``stream``."""
    st = lib().flashbev_sca(ctypes.byref(params), ctypes.c_void_p(stream or 0))
    if check and st != OK:
        raise FlashBevError(st, "flashbev_sca")
    return st


def sca(value, level_hw, lidar2img, offsets, weights, img_hw, bev_range, grid, out=None, hits=None, stream=None,
        chunk_records=0):
    """value: CUDA float32 or bfloat16 [B,N,T,heads,Dh]; offsets [B,Q,heads,L,P,2]; weights [B,Q,heads,L,P] (CUDA float32).
    level_hw: sequence of (H_l, W_l).  Returns CUDA float32 [B, Q, heads*Dh] (marshalling only)."""
    return _result((_native or native()).sca(value, level_hw, lidar2img, offsets, weights, img_hw, bev_range, grid, out, hits,
                                             stream, chunk_records), "flashbev_sca")


def flashbev_workspace_bytes(params: VtParams) -> int:
    return int(lib().flashbev_workspace_bytes(ctypes.byref(params)))


def flashbev_host_staging_bytes(params: VtParams) -> int:
    return int(lib().flashbev_host_staging_bytes(ctypes.byref(params)))


def flashbev_last_launch_count() -> int:
    return int(lib().flashbev_last_launch_count())


def flashbev_last_kernel_name() -> str:
    return lib().flashbev_last_kernel_name().decode()


# ---------------------------------------------------------------------------------------------
# convenience for torch callers (marshalling only)

def sampling_vt(features, lidar2img, img_hw, bev_range, grid, reduce=REDUCE_SUM, out=None,
                valid_count=None, kernel=KERNEL_AUTO, tune=(0, 0, 0, 0), stream=None, layout=NHWC,
                out_dtype=F32, workspace=True):
    """features: CUDA tensor [B,N,Hf,Wf,C] (NHWC) or [B,N,C,Hf,Wf] (NCHW), float32 or bfloat16,
    contiguous; lidar2img: CUDA float32 [B,N,4,4].  Returns the output tensor [B,X,Y,C] (NHWC) or
    [B,C,X,Y] (NCHW), float32 or bfloat16 per ``out_dtype`` (allocated by torch if ``out`` is None).
    ``workspace``: for NCHW tensors and for channel counts that are not whole 16-byte vectors, lend the call the
    scratch ``flashbev_workspace_bytes`` asks for (a torch allocation, or a uint8 CUDA tensor of the caller's);
    False: none, the generic kernel runs.  ``stream``: a raw cudaStream_t instead of the current stream; scratch and a new
    result are allocated for it, and the caller orders the streams."""
    return _result((_native or native()).sampling_vt(features, lidar2img, img_hw, bev_range, grid, reduce, out, valid_count,
                                                     kernel, tune, stream, layout, out_dtype, workspace), "flashbev_sampling_vt")


def sampling_vt_multires(features, lidar2img, img_hw, bev_range, grid, reduce=REDUCE_SUM, out=None,
                         valid_count=None, kernel=KERNEL_AUTO, tune=(0, 0, 0, 0), stream=None, layout=NHWC):
    """features: sequence of CUDA tensors, one per pyramid level, each [B,N,Hf_l,Wf_l,C] (NHWC) or
    [B,N,C,Hf_l,Wf_l] (NCHW) of one dtype.  Returns the float32 sum over the levels (marshalling only)."""
    return _result((_native or native()).sampling_vt_multires(features, lidar2img, img_hw, bev_range, grid, reduce, out,
                                                              valid_count, kernel, tune, stream, layout),
                   "flashbev_sampling_vt_multires")
