"""Builds, in-tree, the C-ABI library (libnpas.so, nvcc for sm_100a) and the CPython extension that the binding's
compute calls go through (_npas_host.so, host code only)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libnpas.so")
HOST_SOURCE = os.path.join(CSRC, "host_ext.cpp")
HOST_LIB = os.path.join(HERE, "_npas_host.so")
SOURCES = ["api.cu", "host_util.cu", "pack.cu", "conv_simt.cu", "linear_simt.cu", "conv_tc.cu", "conv_kr.cu", "conv_stem.cu", "conv_stem_rows.cu", "conv_dn.cu", "conv_d2.cu", "conv_sk.cu", "linear_tc.cu", "linear_dn.cu", "linear_d2.cu", "linear_sk.cu", "linear_two.cu",
           "prune.cu", "static_ws.cu"]


def _stale() -> bool:
    if not os.path.exists(LIB) or not os.path.exists(HOST_LIB):
        return True
    t = min(os.path.getmtime(LIB), os.path.getmtime(HOST_LIB))
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(ROOT, "include", "npas.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def _build_host() -> None:
    import sysconfig
    import torch
    from torch.utils import cpp_extension
    cuda = os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")))
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-DNDEBUG",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-I", sysconfig.get_paths()["include"], "-I", os.path.join(cuda, "include")]
    for d in cpp_extension.include_paths():
        cmd += ["-isystem", d]
    cmd += ["-o", HOST_LIB + ".tmp", HOST_SOURCE]
    for d in cpp_extension.library_paths():
        cmd += ["-L", d]
    cmd += ["-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python", "-L", HERE, "-l:libnpas.so",
            "-Wl,-rpath,$ORIGIN"]
    subprocess.check_call(cmd)
    os.replace(HOST_LIB + ".tmp", HOST_LIB)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "--threads", "0",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB + ".tmp"]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES]
    subprocess.check_call(cmd)
    os.replace(LIB + ".tmp", LIB)
    _build_host()
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
