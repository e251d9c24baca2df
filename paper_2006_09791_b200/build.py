"""Builds libgconv.so with nvcc for sm_100a (cross-compiles without a GPU) and, where there is a C compiler and Python.h, the Python
call module, both in-tree."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "libgconv.so")
CALLS = os.path.join(PKG, "_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))   # (another Python does not load it)
CALLS_SRC = os.path.join(CSRC, "python_calls.c")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17", "-shared",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = _sources() + glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + [
        os.path.join(os.path.dirname(PKG), "include", "gconv.h")]
    return any(os.path.getmtime(p) > t for p in deps)


def build_calls(force: bool = False) -> str:
    """The C module behind gconv.gconv_forward and its like (argument marshalling; no CUDA in it)."""
    if force or not os.path.exists(CALLS) or os.path.getmtime(CALLS_SRC) > os.path.getmtime(CALLS):
        tmp = CALLS + ".tmp.%d" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-shared", "-fPIC", "-I" + sysconfig.get_paths()["include"],
                               "-o", tmp, CALLS_SRC])
        os.replace(tmp, CALLS)
    return CALLS


def build(force: bool = False, verbose: bool = False) -> str:
    if force or _stale():
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
        if verbose:
            flags += ["-Xptxas", "-v"]
        tmp = LIB + ".tmp.%d" % os.getpid()
        cmd = [nvcc] + flags + ["-o", tmp] + _sources()
        subprocess.check_call(cmd)
        os.replace(tmp, LIB)
    try:
        build_calls(force)
    except (OSError, subprocess.CalledProcessError) as e:
        print("the Python call module was not built, calls go through ctypes: %s" % e, file=sys.stderr)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
