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
# the binding's calls, under a name that other interpreters do not load
CALL, CALL_SOURCE = os.path.join(HERE, "_call" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so")), os.path.join(CSRC, "metasd_call.c")
SOURCES = ["metasd_api.cu", "metasd_streaming.cu", "metasd_hinted.cu", "metasd_bulk.cu", "metasd_fused.cu", "metasd_noalloc.cu"]
HEADERS = ["metasd_internal.h", "metasd_device.cuh", "metasd_shapes.h", "metasd_staged.cuh", os.path.join(ROOT, "include", "metasd.h")]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    built = os.path.getmtime(LIB)
    deps = [os.path.join(CSRC, s) for s in SOURCES] + [h if os.path.isabs(h) else os.path.join(CSRC, h) for h in HEADERS]
    return any(os.path.getmtime(d) > built for d in deps)


def build_call(force: bool = False) -> bool:
    """Compile the binding's calls for this interpreter; False where its headers or a compiler are missing (the binding then uses
    ctypes)."""
    include, header = sysconfig.get_paths()["include"], os.path.join(ROOT, "include", "metasd.h")
    untagged = os.path.join(os.path.dirname(CALL), "_call.so")   # an earlier build's, which any interpreter would load
    if untagged != CALL and os.path.exists(untagged):
        os.unlink(untagged)
    if not force and os.path.exists(CALL) and os.path.getmtime(CALL) >= max(os.path.getmtime(f) for f in (CALL_SOURCE, header)):
        return True
    tmp = CALL + ".tmp.%d" % os.getpid()
    try:
        if not os.path.exists(os.path.join(include, "Python.h")):
            raise FileNotFoundError(include)
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-Wall", "-Werror=int-conversion", "-Werror=incompatible-pointer-types",
                               "-shared", "-fPIC", "-I", include, "-I", os.path.dirname(header), CALL_SOURCE, "-o", tmp])
    except FileNotFoundError:
        if os.path.exists(CALL):
            os.unlink(CALL)   # not what the sources say any more
        return False
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
