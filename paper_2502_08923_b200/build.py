"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the Python side of its
search call with the C++ compiler."""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig
import warnings

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcopyspec.so")
HEADER = os.path.join(ROOT, "include", "copyspec.h")
NATIVE_SOURCE = os.path.join(CSRC, "cs_python.cpp")
SOURCES = ["cs_match.cu", "cs_index.cu", "cs_gemm.cu", "cs_gemm_pair.cu", "cs_chain.cu", "cs_small.cu", "cs_layers.cu", "cs_attn.cu", "cs_attn_tc.cu", "cs_attn_tcw.cu", "cs_api.cu", "cs_drafted.cu"]


def native_path() -> str:
    """The search call's Python side.  It goes by the binary interfaces of Python and torch, so a file is named after both."""
    import torch
    return os.path.join(HERE, f"_native.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so")


def _stale(target: str, deps: list) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(p) > os.path.getmtime(target) for p in deps)


def _run(cmd, what):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{what} failed:\n" + res.stderr[-8000:])
    return res.stderr


def _nvcc() -> str:
    return os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")


def _build_native(target: str) -> None:
    import torch
    t = os.path.dirname(torch.__file__)
    cuda = os.path.dirname(os.path.dirname(os.path.realpath(shutil.which(_nvcc()) or _nvcc())))
    part = f"{target}.{os.getpid()}"
    if os.path.exists(target):
        os.remove(target)                # (one of older sources must not stay)
    try:
        _run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
              "-I", os.path.join(t, "include"), "-I", os.path.join(t, "include", "torch", "csrc", "api", "include"),
              "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include"), f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
              NATIVE_SOURCE, "-o", part, "-L", HERE, "-l:libcopyspec.so", "-L", os.path.join(t, "lib"),
              "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], "g++")
        os.replace(part, target)
    finally:
        if os.path.exists(part):
            os.remove(part)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu of the package into libcopyspec.so, and the search call's Python side beside it (only what is missing or older
    than its sources).  That second file is a shorter way to the same function, so it may fail where torch's headers are missing."""
    if force or _stale(LIB, [os.path.join(CSRC, f) for f in os.listdir(CSRC) if not f.endswith(".cpp")] + [HEADER]):
        cmd = [_nvcc(), "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
               "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
               "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
        if verbose:
            cmd.insert(1, "-Xptxas")
            cmd.insert(2, "-v")
        log = _run(cmd, "nvcc")
        if verbose:
            sys.stderr.write(log)
    try:
        native = native_path()
        if force or _stale(native, [NATIVE_SOURCE, HEADER]):
            _build_native(native)
    except (RuntimeError, OSError, ImportError) as e:
        warnings.warn(f"the search call's native side was not built, its general path takes all calls: {e}", RuntimeWarning)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
