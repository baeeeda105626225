"""Builds libdssd.so (the C-ABI CUDA library, nvcc for sm_100a) and _marshal.so (the module through which
binding.py calls it, g++ against torch's headers) in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libdssd.so")
MARSHAL = os.path.join(PKG, "_marshal.so")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    deps = sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh"))
    deps += glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > os.path.getmtime(LIB) for d in deps)


def build_marshal(force: bool = False) -> str:
    """Compile the marshalling module (host code only)."""
    import sysconfig

    src = os.path.join(CSRC, "marshal.cpp")
    deps = [src, os.path.join(ROOT, "include", "dssd.h")]
    if not force and os.path.exists(MARSHAL) and all(os.path.getmtime(d) <= os.path.getmtime(MARSHAL) for d in deps):
        return MARSHAL
    import torch
    from torch.utils import cpp_extension

    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           f"-D_GLIBCXX_USE_CXX11_ABI={int(torch.compiled_with_cxx11_abi())}", "-I", os.path.join(ROOT, "include"),
           "-I", sysconfig.get_paths()["include"], "-o", MARSHAL, src]
    for d in cpp_extension.include_paths(device_type="cuda"):
        cmd += ["-isystem", d]
    for d in cpp_extension.library_paths(device_type="cuda"):
        cmd += ["-L", d]
    cmd += ["-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda", "-ldl"]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if res.returncode != 0:
        sys.stderr.write(res.stdout)
        raise RuntimeError("g++ failed building _marshal.so")
    return MARSHAL


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile both in-tree (nvcc cross-compiles sm_100a without a GPU)."""
    build_marshal(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
           "-o", LIB] + sources()
    if verbose:
        cmd += ["-Xptxas", "-v"]
    res = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed building libdssd.so")
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
