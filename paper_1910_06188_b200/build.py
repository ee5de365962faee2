"""Builds ``libq8.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and ``_q8_native.so`` (the native form of
binding.py's argument marshalling) with g++ against the installed torch.

Usage: ``python -m paper_1910_06188_b200.build [--force] [--verbose]``
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import warnings

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libq8.so")
NATIVE = os.path.join(PKG, "_q8_native.so")

SOURCES = ["q8_api.cu", "q8_attention_sm100.cu", "q8_attention_small_sm100.cu", "q8_elementwise.cu", "q8_gemm_generic.cu", "q8_gemm_sm100.cu", "q8_gemm_splitk_sm100.cu", "q8_hbm_peak.cu", "q8_l2_peak.cu", "q8_mma_peak.cu", "q8_selftest.cu", "q8_static_scratch.cu", "q8_support.cu"]
NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a",
    "-O3", "-std=c++17", "-lineinfo",
    "-Xcompiler", "-fPIC", "-shared",
    "-cudart", "static",
]


def _newest_source_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files += [os.path.join(ROOT, "include", h) for h in ("q8.h", "q8_tools.h")]
    return max(os.path.getmtime(f) for f in files)


def _native_command() -> list:
    import sysconfig

    import torch

    home = os.path.dirname(os.path.abspath(torch.__file__))
    cuda = os.path.dirname(os.path.dirname(shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"))
    include = [os.path.join(home, "include"), os.path.join(home, "include", "torch", "csrc", "api", "include"),
               os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    return [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
            f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", f'-DQ8_TORCH_VERSION="{torch.__version__}"', *("-isystem" + i for i in include),
            "-I", os.path.join(ROOT, "include"), os.path.join(CSRC, "q8_python.cpp"), "-o", NATIVE,
            "-L" + os.path.join(home, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda"]


def _built_for() -> str:
    """What the native marshalling is compiled against, as q8_python.cpp writes it into the module."""
    import torch

    return f"q8 native for torch {torch.__version__}, python {sys.version_info.major}.{sys.version_info.minor}\0"


def _native_is_current() -> bool:
    if not os.path.exists(NATIVE) or os.path.getmtime(NATIVE) < _newest_source_mtime():
        return False
    with open(NATIVE, "rb") as f:
        return _built_for().encode() in f.read()


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile the library and the native marshalling when they are missing or older than any source (or made for
    another torch or Python); returns the library's path.  Without a compiler or headers for the native marshalling, which only makes calls cheaper, the library is all."""
    _build_library(force, verbose)
    if force or not _native_is_current():
        try:
            subprocess.check_call(_native_command())
        except (OSError, subprocess.CalledProcessError) as ex:
            if os.path.exists(NATIVE):
                os.remove(NATIVE)  # made from other sources
            warnings.warn(f"{os.path.basename(NATIVE)} was not built, calls will be marshalled in Python: {ex}", RuntimeWarning)
    return LIB


def _build_library(force: bool, verbose: bool) -> str:
    if not force and os.path.exists(LIB) and os.path.getmtime(LIB) >= _newest_source_mtime():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc, *NVCC_FLAGS, "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += ["-o", LIB] + [os.path.join(CSRC, f) for f in SOURCES]
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
