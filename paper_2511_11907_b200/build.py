"""Builds libkvswap.so (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

Usage:  python -m paper_2511_11907_b200.build [--force]
Objects go to ``_build/`` at the repository root; the shared library lands next to this file, and so does the binding's
extension module where this interpreter's headers are installed (the binding works without it).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
OBJ_DIR = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libkvswap.so")
# the binding's per-layer calls (csrc/pycalls.cpp): an extension module, named for the one interpreter that can load it
CALLS = os.path.join(PKG, "_calls" + (sysconfig.get_config_var("EXT_SUFFIX") or ".so"))

NVCC_FLAGS = ["-O3", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo",
              "-Xcompiler", "-fPIC", "--use_fast_math=false", "-I", INCLUDE, "-I", CSRC]


def _nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found: the kvswap CUDA library cannot be built")
    return exe


def _sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _deps_mtime() -> float:
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return max(os.path.getmtime(f) for f in files)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile every .cu under csrc/ and link libkvswap.so; returns its path."""
    def fresh(f: str) -> bool:
        return not force and os.path.exists(f) and os.path.getmtime(f) >= _deps_mtime()

    if not fresh(LIB):
        _build_library(verbose)
    if not fresh(CALLS):
        _build_calls()
    return LIB


def _build_library(verbose: bool) -> None:
    os.makedirs(OBJ_DIR, exist_ok=True)
    nvcc = _nvcc()
    flags = [f for f in NVCC_FLAGS if f != "--use_fast_math=false"]
    if verbose:
        flags = flags + ["-Xptxas", "-v"]

    def compile_one(src: str) -> str:
        obj = os.path.join(OBJ_DIR, src[:-3] + ".o")
        cmd = [nvcc, *flags, "-c", os.path.join(CSRC, src), "-o", obj]
        res = subprocess.run(cmd, capture_output=True, text=True)
        if res.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{res.stdout}\n{res.stderr}")
        if verbose:
            sys.stderr.write(res.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=min(8, os.cpu_count() or 1)) as ex:
        objs = list(ex.map(compile_one, _sources()))
    cmd = [nvcc, "-shared", "-gencode", "arch=compute_100a,code=sm_100a", "-o", LIB, *objs]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"link failed:\n{res.stdout}\n{res.stderr}")


def _build_calls() -> None:
    headers, gxx = sysconfig.get_paths()["include"], shutil.which("g++")
    if gxx is None or not os.path.exists(os.path.join(headers, "Python.h")):
        return                                   # the binding marshals through ctypes instead
    untagged = os.path.join(PKG, "_calls.so")    # would be loaded by an interpreter without a module of its own
    if untagged != CALLS and os.path.exists(untagged):
        os.remove(untagged)
    cmd = [gxx, "-O2", "-std=c++17", "-shared", "-fPIC", "-I", INCLUDE, "-I", headers,
           os.path.join(CSRC, "pycalls.cpp"), "-o", CALLS]
    res = subprocess.run(cmd, capture_output=True, text=True)
    if res.returncode != 0:
        raise RuntimeError(f"g++ failed on pycalls.cpp:\n{res.stdout}\n{res.stderr}")


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
