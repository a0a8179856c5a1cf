"""Builds libmetasd.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libmetasd.so")
CALL, CALL_SOURCE = os.path.join(HERE, "_call.so"), os.path.join(CSRC, "metasd_call.c")   # the binding's calls
SOURCES = ["metasd_api.cu", "metasd_streaming.cu", "metasd_hinted.cu", "metasd_bulk.cu", "metasd_fused.cu", "metasd_noalloc.cu"]
HEADERS = ["metasd_internal.h", "metasd_device.cuh", "metasd_staged.cuh", os.path.join(ROOT, "include", "metasd.h")]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    built = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + [h if os.path.isabs(h) else os.path.join(CSRC, h) for h in HEADERS]
    return any(os.path.getmtime(d) > built for d in deps)


def build_call(force: bool = False) -> bool:
    """Compile the binding's calls for this interpreter; False where its headers are missing (the binding then uses ctypes)."""
    include = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(include, "Python.h")):
        return False
    if force or not os.path.exists(CALL) or os.path.getmtime(CALL_SOURCE) > os.path.getmtime(CALL):
        tmp = CALL + ".tmp.%d" % os.getpid()
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-shared", "-fPIC", "-I", include,
                               "-I", os.path.join(ROOT, "include"), CALL_SOURCE, "-o", tmp])
        os.replace(tmp, CALL)
    return True


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu for sm_100a into one shared library, and the binding's calls; returns the library's path."""
    build_call(force)
    if not force and not _stale():
        return LIB
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB + ".tmp.%d" % os.getpid()
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-Xcompiler", "-fPIC", "-shared", "-cudart", "static", "-t", "4",
           "-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
