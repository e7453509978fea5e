"""Builds libonnx_b200.so in-tree with nvcc for sm_100a, and the binding's native call path with g++.

Usage: ``python -m paper_2008_08272_b200.build [--force] [--verbose]``.  The library needs nvcc alone; the native call
path also needs torch's headers, and where it cannot be built the binding makes its calls through ctypes.
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB_DIR = os.path.join(HERE, "_lib")
LIB_PATH = os.path.join(LIB_DIR, "libonnx_b200.so")
EXT_SRC = os.path.join(HERE, "ext", "fast_binding.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "--threads", "0",
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")) + glob.glob(os.path.join(CSRC, "*.cpp")))


def _inputs():
    return sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))


def is_stale() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    t = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(f) > t for f in _inputs())


def ext_path() -> str:
    """The native call path's file.  It calls into torch's C++ libraries and into CPython, neither of which keeps its ABI, so
    their versions are part of the name: a file built for others is never loaded."""
    import importlib.metadata
    return os.path.join(LIB_DIR, "_onnxb_fast.%s.torch-%s.so" % (sys.implementation.cache_tag, importlib.metadata.version("torch")))


def build_ext(force: bool = False, verbose: bool = False) -> str:
    """Compile the binding's native call path (a CPython extension on torch's C++ tensors)."""
    import sysconfig
    path = ext_path()
    deps = [EXT_SRC, os.path.join(ROOT, "include", "onnx_b200.h")]
    if not force and os.path.exists(path) and all(os.path.getmtime(path) >= os.path.getmtime(f) for f in deps):
        return path
    import torch
    tdir = os.path.dirname(torch.__file__)
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    os.makedirs(LIB_DIR, exist_ok=True)
    tmp = path + ".%d.tmp" % os.getpid()
    cmd = ["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-D_GLIBCXX_USE_CXX11_ABI=%d" % int(torch._C._GLIBCXX_USE_CXX11_ABI),
           "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(tdir, "include"),
           "-I" + os.path.join(tdir, "include", "torch", "csrc", "api", "include"),
           "-I" + os.path.join(cuda, "include"), "-I" + sysconfig.get_paths()["include"], EXT_SRC, "-o", tmp,
           "-L" + os.path.join(tdir, "lib"), "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_cuda", "-ltorch_python", "-ldl"]
    proc = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout)
    if proc.returncode != 0:
        raise RuntimeError("g++ failed building " + os.path.basename(path))
    os.replace(tmp, path)
    return path


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every CUDA source of the library into one shared object."""
    if not force and not is_stale():
        return LIB_PATH
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    os.makedirs(LIB_DIR, exist_ok=True)
    tmp = LIB_PATH + ".%d.tmp" % os.getpid()
    cmd = [nvcc] + NVCC_FLAGS + ["-I" + os.path.join(ROOT, "include"), "-I" + CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += os.environ.get("ONNXB_NVCC_EXTRA", "").split()
    cmd += sources() + ["-o", tmp]
    proc = subprocess.run(cmd, stdout=subprocess.PIPE, stderr=subprocess.STDOUT, text=True)
    if verbose or proc.returncode != 0:
        sys.stderr.write(proc.stdout)
    if proc.returncode != 0:
        raise RuntimeError("nvcc failed building libonnx_b200.so")
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    flags = dict(force="--force" in sys.argv, verbose="--verbose" in sys.argv)
    print(build(**flags))
    try:
        print(build_ext(**flags))
    except Exception as e:
        print("the binding's native call path was not built (%s): it will call through ctypes" % e, file=sys.stderr)
