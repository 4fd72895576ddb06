"""Build the CUDA library in-tree for sm_100a (nvcc cross-compiles without a GPU) and its CPython entry points."""
from __future__ import annotations

import importlib.metadata
import importlib.util
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(_HERE)
SOURCES = [os.path.join(_HERE, "csrc", "flashbev.cu")]
HEADERS = [os.path.join(ROOT, "include", "flashbev.h"), os.path.join(_HERE, "csrc", "vt_tiled.cuh"),
           os.path.join(_HERE, "csrc", "vt_backward.cuh")]
LIB = os.path.join(_HERE, "libflashbev.so")

NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include")]


LIB_DEBUG_BOUNDS = os.path.join(_HERE, "libflashbev_debug_bounds.so")


NATIVE_SOURCES = [os.path.join(_HERE, "csrc", "native.cpp")]
NATIVE = os.path.join(_HERE, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_RECORD = os.path.join(_HERE, "_native.built_with")  # what NATIVE was built with


def needs_build(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    return any(os.path.getmtime(s) > t for s in SOURCES + HEADERS)


def native_prerequisites() -> str | None:
    """What the extension module needs and this machine lacks (None: nothing).  The library itself needs none of it."""
    spec = importlib.util.find_spec("torch")
    if spec is None or not spec.submodule_search_locations:
        return "PyTorch is not installed"
    if not os.path.exists(os.path.join(spec.submodule_search_locations[0], "lib", "libc10_cuda.so")):
        return "the installed PyTorch has no CUDA part"
    if not os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h")):
        return "the headers of Python are not installed"
    return None


def _built_with() -> str:
    """What the extension module is bound to beside its sources: it calls PyTorch's C++ libraries, whose classes and symbols
    change from version to version."""
    return f"torch {importlib.metadata.version('torch')}\n"


def needs_native_build() -> bool:
    if not os.path.exists(NATIVE) or not os.path.exists(NATIVE_RECORD):
        return True
    with open(NATIVE_RECORD) as f:
        if f.read() != _built_with():
            return True
    return any(os.path.getmtime(s) > os.path.getmtime(NATIVE) for s in NATIVE_SOURCES + HEADERS[:1])


def build_native(force: bool = False) -> str:
    """Compile csrc/native.cpp (g++, PyTorch headers) into the extension module next to this file; returns its path."""
    missing = native_prerequisites()
    if missing:
        raise RuntimeError(f"the extension module for torch tensors cannot be built: {missing}")
    if force or needs_native_build():
        torch_dir = importlib.util.find_spec("torch").submodule_search_locations[0]
        inc = [os.path.join(torch_dir, "include"), os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"),
               sysconfig.get_paths()["include"], "/usr/local/cuda/include", os.path.join(ROOT, "include")]
        cmd = ([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden", "-w"] +
               [f"-I{d}" for d in inc] + NATIVE_SOURCES +
               [f"-L{os.path.join(torch_dir, 'lib')}", "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
                f"-L{_HERE}", "-lflashbev", "-Wl,-rpath,$ORIGIN", "-o", NATIVE])
        subprocess.run(cmd, check=True)
        with open(NATIVE_RECORD, "w") as f:
            f.write(_built_with())
    return NATIVE


def build(force: bool = False, verbose: bool = False, debug_bounds: bool = False) -> str:
    """Compile csrc/*.cu into libflashbev.so next to this file, and the extension module over it where PyTorch is installed;
    returns the library's path.

    ``debug_bounds``: build libflashbev_debug_bounds.so instead, with -DFLASHBEV_DEBUG_BOUNDS: every index the
    tiled kernel computes is range-checked, violations are counted into the caller's ``debug_error_word`` and
    the access is redirected to a safe slot (the stand-in for a memory checker on machines where none may run)."""
    lib = LIB_DEBUG_BOUNDS if debug_bounds else LIB
    if force or needs_build(lib):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = ([nvcc] + NVCC_FLAGS + (["-DFLASHBEV_DEBUG_BOUNDS"] if debug_bounds else []) +
               (["-Xptxas", "-v"] if verbose else []) + SOURCES + ["-o", lib])
        subprocess.run(cmd, check=True)
    if not debug_bounds:
        missing = native_prerequisites()
        if missing:  # the C ABI and its ctypes mirror work without; calls with torch tensors raise ImportError
            print(f"libflashbev.so only, no extension module for torch tensors: {missing}", file=sys.stderr)
        else:
            build_native(force)
    return lib


if __name__ == "__main__":
    print(build(force=True, verbose=True))
