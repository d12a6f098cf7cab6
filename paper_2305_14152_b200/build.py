"""Build the sm_100a shared library in-tree with nvcc (no GPU needed to compile)."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libpeqa_b200.so")
NATIVE_SRC = os.path.join(CSRC, "pybinding.cpp")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-shared", "-Xptxas", "-v",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def native_path() -> str:
    """The extension module for this interpreter and this torch: both are in its name, so that a file
    built for others is never loaded."""
    import torch
    return os.path.join(HERE, f"_native.{sysconfig.get_config_var('SOABI')}.torch-{torch.__version__}.so")


def _native_prerequisite():
    """What the extension module needs and this machine lacks, or None."""
    try:
        import torch
    except ImportError:
        return "torch"
    if not os.path.exists(os.path.join(sysconfig.get_paths()["include"], "Python.h")):
        return "Python.h"
    if not os.path.exists(os.path.join(os.path.dirname(torch.__file__), "include", "ATen", "ATen.h")):
        return "the headers of torch"
    if shutil.which(os.environ.get("CXX", "g++")) is None:
        return "a C++ compiler"
    return None


def _build_native(verbose: bool) -> None:
    """The extension module that marshals the frequent calls (binding.py)."""
    import torch
    base = os.path.dirname(os.path.abspath(torch.__file__))
    libs = os.path.join(base, "lib")
    cmd = [os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-fPIC", "-shared", "-fvisibility=hidden",
           "-I", os.path.join(ROOT, "include"), "-I", os.path.join(base, "include"),
           "-I", os.path.join(base, "include", "torch", "csrc", "api", "include"),
           "-I", sysconfig.get_paths()["include"], "-I", "/usr/local/cuda/include",
           NATIVE_SRC, "-o", native_path(), "-L", libs, "-ltorch_python", "-ltorch", "-ltorch_cpu", "-lc10", "-lc10_cuda",
           "-L", HERE, "-lpeqa_b200", "-Wl,-rpath,$ORIGIN", "-Wl,-rpath," + libs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or res.returncode != 0:
        sys.stderr.write(res.stdout + res.stderr)
    if res.returncode != 0:
        raise RuntimeError(f"building {native_path()} failed")


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + ["-o", LIB] + sources()
        res = subprocess.run(cmd, capture_output=True, text=True)
        if verbose or res.returncode != 0:
            sys.stderr.write(res.stdout + res.stderr)
        if res.returncode != 0:
            raise RuntimeError("nvcc failed building libpeqa_b200.so")
    # A program that calls the C ABI needs no more than this.  The binding does, and says so at its first call.
    missing = _native_prerequisite()
    if missing is not None:
        sys.stderr.write(f"paper_2305_14152_b200: the extension module of the binding is not built, {missing} is missing\n")
        return LIB
    native = native_path()
    header = os.path.join(ROOT, "include", "peqa.h")
    if force or not os.path.exists(native) or \
            os.path.getmtime(native) < max(os.path.getmtime(NATIVE_SRC), os.path.getmtime(header)):
        _build_native(verbose)
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
