"""Builds the CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the Python side of its
search call with the C++ compiler."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libcopyspec.so")
NATIVE = os.path.join(HERE, "_native.so")
SOURCES = ["cs_match.cu", "cs_index.cu", "cs_gemm.cu", "cs_gemm_pair.cu", "cs_chain.cu", "cs_small.cu", "cs_layers.cu", "cs_attn.cu", "cs_attn_tc.cu", "cs_attn_tcw.cu", "cs_api.cu", "cs_drafted.cu"]


def _newer_than_lib() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(NATIVE):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(NATIVE))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "copyspec.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def _run(cmd, what):
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"{what} failed:\n" + res.stderr[-8000:])
    return res.stderr


def _build_native() -> None:
    import torch
    t = os.path.dirname(torch.__file__)
    _run([os.environ.get("CXX", "g++"), "-std=c++17", "-O2", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"),
          "-I", os.path.join(t, "include"), "-I", os.path.join(t, "include", "torch", "csrc", "api", "include"),
          "-I", sysconfig.get_paths()["include"], "-I", "/usr/local/cuda/include", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
          os.path.join(CSRC, "cs_python.cpp"), "-o", NATIVE, "-L", HERE, "-l:libcopyspec.so", "-L", os.path.join(t, "lib"),
          "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-Wl,-rpath,$ORIGIN"], "g++")


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu of the package into libcopyspec.so, and _native.so beside it (only when sources changed)."""
    if not force and not _newer_than_lib():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-std=c++17", "-O3", "-lineinfo", "-gencode", "arch=compute_100a,code=sm_100a",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    log = _run(cmd, "nvcc")
    if verbose:
        sys.stderr.write(log)
    _build_native()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
