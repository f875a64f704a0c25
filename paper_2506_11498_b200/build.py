"""Builds the CUDA library in-tree with nvcc for sm_100a (no JIT cache, no torch extension)."""
from __future__ import annotations

import glob
import importlib.machinery
import os
import subprocess
import sys
import sysconfig

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "liblrsa.so")
# Python module over two of the library's calls, for the interpreter that builds it.  The binding works without it.
CALL = os.path.join(_HERE, "_lrsa_call" + importlib.machinery.EXTENSION_SUFFIXES[0])
NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "-shared"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _older(target, deps) -> bool:
    return not os.path.exists(target) or any(os.path.getmtime(f) > os.path.getmtime(target) for f in deps)


def _abi():
    return glob.glob(os.path.join(_HERE, "..", "include", "*.h"))


def is_stale() -> bool:
    return _older(LIB, sources() + glob.glob(os.path.join(CSRC, "*.h")) + _abi())


def call_is_stale() -> bool:
    return _older(CALL, [os.path.join(CSRC, "pycall.c")] + _abi())


def build_call() -> bool:
    """Compiles the helper module.  Where that is not possible (no compiler, no Python.h) none is left behind: an older one
    would call the library with the interface it was built for."""
    cmd = [os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], "-o", CALL,
           os.path.join(CSRC, "pycall.c"), "-L", _HERE, "-l:liblrsa.so", "-Wl,-rpath,$ORIGIN"]
    if os.path.exists(CALL):
        os.remove(CALL)
    try:
        subprocess.check_call(cmd)
    except (OSError, subprocess.CalledProcessError) as e:
        print(f"{os.path.basename(CALL)} was not built ({e}): its calls go through ctypes", file=sys.stderr)
        return False
    return True


def build(force: bool = False, verbose: bool = False) -> str:
    if force or is_stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + sources()
        subprocess.check_call(cmd)
    if force or call_is_stale():
        build_call()
    return LIB


if __name__ == "__main__":
    print(build(force=True, verbose=True))
