"""Builds libquantpipe.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a, and _qpcall.so (the
Python call path into it) with the C compiler.

    python -m paper_2211_04515_b200.build [--force] [--verbose] [--check]
"""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
LIB = os.path.join(PKG, "libquantpipe.so")
LIB_CHECK = os.path.join(PKG, "libquantpipe_check.so")    # the same sources with -DQP_CHECK_BOUNDS

CALL_SRC = os.path.join(CSRC, "qp_call.c")
CALL_LIB = os.path.join(PKG, "_qpcall.so")

NVCC_FLAGS = [
    "-shared", "-Xcompiler", "-fPIC", "-std=c++17", "-O3", "-lineinfo",
    "--fmad=false",                                    # fused multiply-adds only where the code writes fma()
    "-gencode", "arch=compute_100a,code=sm_100a",
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; set NVCC or put the CUDA toolkit on PATH")


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def is_stale(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(INCLUDE, "*.h"))
    return any(os.path.getmtime(d) > t for d in deps)


def build_call_path(force: bool = False) -> str:
    """Builds the extension module that carries calls from Python into the library."""
    if not force and os.path.exists(CALL_LIB) and os.path.getmtime(CALL_LIB) >= os.path.getmtime(CALL_SRC):
        return CALL_LIB
    tmp = CALL_LIB + f".tmp{os.getpid()}"
    subprocess.run([os.environ.get("CC", "gcc"), "-shared", "-fPIC", "-O2", "-Wall", "-I", sysconfig.get_paths()["include"],
                    "-o", tmp, CALL_SRC], check=True)
    os.replace(tmp, CALL_LIB)
    return CALL_LIB


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    """Builds the library; check=True builds the variant with index checks (libquantpipe_check.so)."""
    build_call_path(force)
    lib = LIB_CHECK if check else LIB
    if not force and not is_stale(lib):
        return lib
    tmp = lib + f".tmp{os.getpid()}"
    cmd = [_nvcc(), "-t", str(min(8, os.cpu_count() or 1)), *NVCC_FLAGS, *(["-DQP_CHECK_BOUNDS"] if check else []), "-I", INCLUDE, "-I", CSRC, "-o", tmp, *sources()]
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
        print(" ".join(cmd))
    subprocess.run(cmd, check=True)
    os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, check="--check" in sys.argv))
