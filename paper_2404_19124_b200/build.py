"""Builds libspec_b200.so in-tree with nvcc for sm_100a (no JIT cache, no torch extension), and beside it the CPython module
_pycall that marshals the calls of a decoding step (the binding does without where the interpreter's headers or a C compiler
are missing).  That module is compiled against one interpreter's object layout, so its file name carries the interpreter's
tag and no other interpreter imports it."""
from __future__ import annotations

import os
import subprocess
import sys
import sysconfig
import warnings

_PKG = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_PKG)
CSRC = os.path.join(_PKG, "csrc")
INCLUDE = os.path.join(_ROOT, "include")
LIB_PATH = os.path.join(_PKG, "libspec_b200.so")
PYCALL_PATH = os.path.join(_PKG, "_pycall" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))
SOURCES = ["spec_api.cu", "verify_kernels.cu", "draft_kernels.cu", "draft_small.cu", "fp8_kernels.cu", "gemm_tcgen05.cu",
           "gemm_pair.cu", "gemm_simt.cu"]


def _newest_source_mtime() -> float:
    paths = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "spec_b200.h")]
    return max(os.path.getmtime(p) for p in paths)


def _remove(path: str) -> None:
    if os.path.exists(path):
        os.remove(path)


def _build_pycall(force: bool) -> None:
    source = os.path.join(CSRC, "pycall.c")
    newest = max(os.path.getmtime(source), os.path.getmtime(os.path.join(INCLUDE, "spec_b200.h")))
    untagged = os.path.join(_PKG, "_pycall.so")      # any interpreter would import it
    if untagged != PYCALL_PATH:
        _remove(untagged)
    if not force and os.path.exists(PYCALL_PATH) and os.path.getmtime(PYCALL_PATH) >= newest:
        return
    _remove(PYCALL_PATH)                              # nothing rather than a module of another source
    headers = sysconfig.get_paths()["include"]
    if not os.path.exists(os.path.join(headers, "Python.h")):
        return
    tmp = PYCALL_PATH + f".tmp{os.getpid()}"
    try:
        subprocess.check_call([os.environ.get("CC", "gcc"), "-O2", "-std=c11", "-Wall", "-shared", "-fPIC", "-I", headers,
                               "-I", INCLUDE, source, "-o", tmp])
    except (OSError, subprocess.CalledProcessError) as e:
        _remove(tmp)
        warnings.warn(f"_pycall was not built, calls are marshalled in Python: {e}")
        return
    os.replace(tmp, PYCALL_PATH)


def build(force: bool = False, verbose: bool = False) -> str:
    _build_pycall(force)
    if not force and os.path.exists(LIB_PATH) and os.path.getmtime(LIB_PATH) >= _newest_source_mtime():
        return LIB_PATH
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    tmp = LIB_PATH + f".tmp{os.getpid()}"
    cmd = [nvcc, "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-cudart", "static", "-I", INCLUDE, "-I", CSRC]
    if verbose:
        cmd += ["-Xptxas", "-v"]
    cmd += [os.path.join(CSRC, s) for s in SOURCES] + ["-o", tmp]
    subprocess.check_call(cmd)
    os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
