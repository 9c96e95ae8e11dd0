"""Build libtt.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and the CPython module of its hot calls."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libtt.so")
SOURCES = ["tt_host.cpp", "tt_kernels.cu", "tt_conv.cu", "tt_attention.cu", "tt_device.cu"]
HEADERS = [os.path.join(CSRC, "tt_internal.h"), os.path.join(CSRC, "tt_ptx.cuh"), os.path.join(ROOT, "include", "tt.h")]
CALL_LIB = os.path.join(HERE, "_ttcall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
CALL_SOURCE = os.path.join(CSRC, "tt_pycall.cpp")


def _stale(target, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def needs_build() -> bool:
    return _stale(LIB, [os.path.join(CSRC, s) for s in SOURCES] + HEADERS) or _stale(CALL_LIB, [CALL_SOURCE, HEADERS[-1]])


def build(force: bool = False, verbose: bool = False) -> str:
    inc = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    if force or _stale(LIB, [os.path.join(CSRC, s) for s in SOURCES] + HEADERS):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        cmd = [nvcc, "-shared", "-o", LIB, "-std=c++17", "-O3", "-lineinfo", "--threads", "0",
               "-gencode", "arch=compute_100a,code=sm_100a",
               "-Xcompiler", "-fPIC,-Wall,-Wno-unused-function", "-cudart", "static"] + inc
        if verbose:
            cmd += ["-Xptxas", "-v"]
        subprocess.check_call(cmd + [os.path.join(CSRC, s) for s in SOURCES])
    if force or _stale(CALL_LIB, [CALL_SOURCE, HEADERS[-1]]):
        subprocess.check_call(["g++", "-shared", "-fPIC", "-O2", "-std=c++17", "-Wall", "-o", CALL_LIB] + inc +
                              ["-I", sysconfig.get_paths()["include"], CALL_SOURCE])
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
