"""Builds libsdq_b200.so (nvcc for sm_100a, cross-compiles without a GPU) and the binding's native half (g++) in-tree."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

import torch

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libsdq_b200.so")
# C++ against torch's headers: the versions it was built for are part of the name, so a module of another torch is never loaded
BINDING = os.path.join(_HERE, "_binding-%s-torch%s.so" % (sys.implementation.cache_tag, torch.__version__))
BINDING_SOURCE = "sdq_python.cpp"
SOURCES = ["sdq_api.cu", "sdq_pack.cu", "sdq_quant_act.cu", "sdq_linear.cu", "sdq_linear_pair.cu", "sdq_linear_group.cu", "sdq_plain.cu", "sdq_calib.cu", "sdq_diag.cu"]
HEADERS = ["sdq_internal.h", "sdq_layout.h", "sdq_linear.h", "sdq_plain.h", "sdq_ptx.cuh", "sdq_codec.cuh", os.path.join("..", "..", "include", "sdq.h"), os.path.join("..", "..", "include", "sdq_diag.h")]
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-shared",
              "-Xcompiler", "-fPIC"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(os.path.join(CSRC, f)) > t for f in SOURCES + HEADERS)


def _binding_stale() -> bool:
    if not os.path.exists(BINDING):
        return True
    t = os.path.getmtime(BINDING)
    return any(os.path.getmtime(os.path.join(CSRC, f)) > t for f in [BINDING_SOURCE, os.path.join("..", "..", "include", "sdq.h")])


def _build_binding() -> None:
    root = os.path.dirname(torch.__file__)
    inc = [os.path.join(root, "include"), os.path.join(root, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
           os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")]
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)] + ["-I" + i for i in inc]
    # torch's own libraries are in the process already (the package imports torch first); libsdq_b200.so sits beside this file
    cmd += ["-o", BINDING + ".tmp", BINDING_SOURCE, "-L" + os.path.join(root, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10", "-lc10_cuda",
            "-L" + _HERE, "-l:libsdq_b200.so", "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd, cwd=CSRC)
    os.replace(BINDING + ".tmp", BINDING)


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB + ".tmp"] + SOURCES
        subprocess.check_call(cmd, cwd=CSRC)
        os.replace(LIB + ".tmp", LIB)
    if force or _binding_stale():
        try:
            _build_binding()
        except (OSError, subprocess.CalledProcessError) as e:
            warnings.warn("the binding's native half was not built (%s): calls go through ctypes, 6 to 12 us slower each" % e)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
