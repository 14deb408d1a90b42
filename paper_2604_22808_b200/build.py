"""Builds the CUDA library in-tree for sm_100a: `python -m paper_2604_22808_b200.build`."""
from __future__ import annotations

import glob
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
LIB = os.path.join(PKG, "libfreqformer.so")
LIB_DEBUG = os.path.join(PKG, "libfreqformer_debug.so")     # the same sources with -DFF_DEBUG (device-side range checks)
LIB_CLOCKS = os.path.join(PKG, "libfreqformer_clocks.so")   # ... with -DFF_CLOCKS (cycle sums, see clocks.py)


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found; the FreqFormer CUDA library cannot be built")


def sources():
    return sorted(glob.glob(os.path.join(PKG, "csrc", "*.cu")))


def needs_build(lib: str = LIB) -> bool:
    if not os.path.exists(lib):
        return True
    t = os.path.getmtime(lib)
    deps = sources() + glob.glob(os.path.join(PKG, "csrc", "*.h")) + glob.glob(os.path.join(PKG, "csrc", "*.cuh")) \
        + glob.glob(os.path.join(ROOT, "include", "*.h"))
    return any(os.path.getmtime(f) > t for f in deps)


def build(force: bool = False, verbose: bool = False, debug: bool = False, clocks: bool = False) -> str:
    lib = LIB_CLOCKS if clocks else (LIB_DEBUG if debug else LIB)
    if not force and not needs_build(lib):
        return lib
    cmd = [_nvcc(), "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
           "-shared", "-Xcompiler", "-fPIC", "-I", os.path.join(ROOT, "include"), "-I", os.path.join(PKG, "csrc"),
           "-o", lib] + (["-DFF_CLOCKS"] if clocks else ["-DFF_DEBUG"] if debug else []) + sources()
    cmd[1:1] = os.environ.get("FF_NVCC_FLAGS", "").split()      # e.g. --threads 8
    if verbose:
        cmd.insert(1, "-Xptxas")
        cmd.insert(2, "-v")
    res = subprocess.run(cmd, capture_output=True, text=True)
    if verbose:
        sys.stderr.write(res.stderr)
    if res.returncode != 0:
        raise RuntimeError("nvcc failed:\n" + res.stdout + res.stderr)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv, debug="--debug" in sys.argv,
                clocks="--clocks" in sys.argv))
