"""Build libdropit.so (CUDA kernels + C ABI, nvcc for sm_100a) and _native.so (its torch binding, g++) in-tree."""
from __future__ import annotations

import glob
import importlib.util
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libdropit.so")
NATIVE = os.path.join(PKG, "_native.so")
NATIVE_SRC = os.path.join(CSRC, "native.cpp")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(CSRC, "*.h")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ into one shared library; returns its path."""
    if not force and not _stale():
        _build_native(force)
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-shared",
           "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", CSRC, "-o", tmp] + sources()
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    subprocess.run(cmd, check=True)
    os.replace(tmp, LIB)
    _build_native(True)
    return LIB


def _build_native(force: bool):
    """Compile the torch binding against the installed torch's headers and link it to libdropit.so beside it."""
    deps = [NATIVE_SRC, os.path.join(CSRC, "layer_ops.h"), os.path.join(ROOT, "include", "dropit.h"),
            os.path.join(os.path.dirname(importlib.util.find_spec("torch").origin), "version.py")]     # another torch, another ABI
    if not force and os.path.exists(NATIVE) and os.path.getmtime(NATIVE) > max(os.path.getmtime(d) for d in deps):
        return
    import torch

    tdir = os.path.dirname(torch.__file__)
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc"))), "include")
    includes = [os.path.join(ROOT, "include"), CSRC, os.path.join(tdir, "include"),
                os.path.join(tdir, "include", "torch", "csrc", "api", "include"), cuda, sysconfig.get_path("include")]
    tmp = NATIVE + ".tmp.%d" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-DTORCH_API_INCLUDE_EXTENSION_H",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI)]
    cmd += [a for i in includes for a in ("-I", i)]
    cmd += [NATIVE_SRC, "-o", tmp, "-L", PKG, "-l:libdropit.so", "-Wl,-rpath,$ORIGIN", "-L", os.path.join(tdir, "lib"),
            "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch", "-ltorch_python"]
    subprocess.run(cmd, check=True)
    os.replace(tmp, NATIVE)


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
