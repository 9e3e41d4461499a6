"""Builds the C-ABI CUDA library in-tree with nvcc for sm_100a (cross-compiles without a GPU), and the CPython module
that passes tensors to it."""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
LIB = os.path.join(PKG, "librmuscle.so")
MODULE = os.path.join(PKG, "_rmuscle.so")
MODULE_SRC = os.path.join(CSRC, "rm_python.cpp")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "--expt-relaxed-constexpr", "--extended-lambda", "-Xcompiler", "-fPIC"]


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def _run(cmd, what: str, verbose: bool = False) -> None:
    r = subprocess.run(cmd, capture_output=True, text=True)
    if verbose or r.returncode != 0:
        sys.stderr.write(r.stdout + r.stderr)
    if r.returncode != 0:
        raise RuntimeError(f"building {what} failed")


def build_library(force: bool = False, verbose: bool = False) -> str:
    headers = glob.glob(os.path.join(CSRC, "*.cuh")) + glob.glob(os.path.join(ROOT, "include", "*.h"))
    inc = ["-I", os.path.join(ROOT, "include"), "-I", CSRC]
    tmp = f".tmp{os.getpid()}"
    if force or _stale(LIB, sources() + headers):
        nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
        flags = NVCC_FLAGS + os.environ.get("RM_EXTRA_NVCC_FLAGS", "").split() + (["-Xptxas", "-v"] if verbose else [])
        objs = [(src, f"{LIB}{tmp}.{i}.o") for i, src in enumerate(sources())]
        try:
            with ThreadPoolExecutor(max_workers=min(len(objs), os.cpu_count() or 1)) as ex:
                list(ex.map(lambda o: _run([nvcc, *flags, *inc, "-c", "-o", o[1], o[0]], os.path.basename(o[0]), verbose), objs))
            _run([nvcc, *NVCC_FLAGS, "-shared", "-o", LIB + tmp, *[o for _, o in objs]], "librmuscle.so", verbose)
        finally:
            for _, o in objs:
                if os.path.exists(o):
                    os.remove(o)
        os.replace(LIB + tmp, LIB)
    if force or _stale(MODULE, [MODULE_SRC] + headers):
        _run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-shared", "-fPIC", "-I", sysconfig.get_paths()["include"], *inc,
              "-o", MODULE + tmp, MODULE_SRC, "-L", PKG, "-l:librmuscle.so", "-Wl,-rpath,$ORIGIN"], "_rmuscle.so", verbose)
        os.replace(MODULE + tmp, MODULE)
    return LIB


if __name__ == "__main__":
    print(build_library(force=True, verbose="-v" in sys.argv))
