"""Builds the CUDA shared library in-tree with nvcc for sm_100a, and the native half of the Python binding with g++.

    python -m paper_2607_23815_b200.build          # (re)build if sources are newer
    python -m paper_2607_23815_b200.build --force
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libkvattn.so")
BINDING = os.path.join(HERE, "_kvattn_native.so")
BINDING_FOR = os.path.join(HERE, "_kvattn_native.torch")  # what the module was compiled against (see binding_abi)
SOURCES = ["pool.cu", "attn_small.cu", "attn_decode.cu", "attn_extend_tc.cu", "attn_decode_static.cu", "attn_shared.cu", "selftest.cu", "api.cu"]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--shared", "-Xcompiler", "-fPIC", "-Xptxas", "-v"]


def _nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is needed to build libkvattn.so")


def _stale(target: str, suffixes) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(suffixes)] + [os.path.join(HERE, "..", "include", "kvattn.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, verbose: bool, what: str) -> None:
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"building {what} failed")


def binding_abi() -> str:
    """The module uses torch's C++ classes and Python's C API: one compiled against other versions must not be loaded."""
    import torch
    return f"torch {torch.__version__} {sysconfig.get_config_var('SOABI')}"


def binding_made_for() -> str:
    """What the module that is there was compiled against, "" if that is not known (the module was copied alone)."""
    try:
        with open(BINDING_FOR) as f:
            return f.read()
    except OSError:
        return ""


def build_binding(force: bool = False, verbose: bool = False) -> str:
    """The extension module that unpacks torch tensors and calls libkvattn.so (which lies beside it)."""
    if not force and binding_made_for() == binding_abi() and not _stale(BINDING, (".cpp",)):
        return BINDING
    import torch
    from torch.utils import cpp_extension as ext
    libs = os.path.join(os.path.dirname(torch.__file__), "lib")
    cuda = os.path.dirname(os.path.dirname(_nvcc()))
    inc = ext.include_paths() + [os.path.join(cuda, "include"), sysconfig.get_paths()["include"]]
    _run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}"]
         + [f"-I{d}" for d in inc] + [os.path.join(CSRC, "binding.cpp"), "-o", BINDING, LIB, "-Wl,-rpath,$ORIGIN", f"-L{libs}",
                                      "-lc10", "-lc10_cuda", "-ltorch", "-ltorch_cpu", "-ltorch_python"], verbose, "_kvattn_native.so")
    with open(BINDING_FOR, "w") as f:
        f.write(binding_abi())
    return BINDING


def build_library(force: bool = False, verbose: bool = False) -> str:
    if force or _stale(LIB, (".cu", ".cuh", ".h")):
        _run([_nvcc()] + NVCC_FLAGS + ["-Xlinker", "-soname=libkvattn.so", "-o", LIB] + [os.path.join(CSRC, s) for s in SOURCES],
             verbose, "libkvattn.so")
    build_binding(force, verbose)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose=True))
