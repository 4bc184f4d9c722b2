"""Builds libckv.so (sm_100a) next to this file with nvcc, and with the host compiler the CPython helper _pycall.so
of the binding.  No GPU is needed to build.

    python paper_2601_19178_b200/build.py [--force] [--verbose] [--bounds]     (or: python __graft_entry__.py)
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys
import sysconfig

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libckv.so")
PYCALL = os.path.join(PKG, "_pycall.so")
LIB_BOUNDS = os.path.join(PKG, "libckv_bounds.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-Xcompiler", "-fvisibility=hidden",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    raise RuntimeError("nvcc not found")


def _newest(paths) -> float:
    return max(os.path.getmtime(p) for p in paths)


def build_pycall(force: bool = False) -> str:
    src = os.path.join(CSRC, "pycall.c")
    if force or not os.path.exists(PYCALL) or os.path.getmtime(PYCALL) < os.path.getmtime(src):
        tmp = PYCALL + f".tmp{os.getpid()}"
        cmd = [os.environ.get("CC") or "gcc", "-O2", "-Wall", "-shared", "-fPIC", "-fvisibility=hidden",
               "-I", sysconfig.get_paths()["include"], src, "-o", tmp]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("the host compiler failed on " + src)
        os.replace(tmp, PYCALL)
    return PYCALL


def build(force: bool = False, verbose: bool = False, bounds: bool = False) -> str:
    """bounds=True builds libckv_bounds.so instead: the same library with every index, row and shared-memory
    offset the kernels compute range-checked into the context's error word (-DCKV_BOUNDS)."""
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = glob.glob(os.path.join(CSRC, "*.h")) + glob.glob(os.path.join(CSRC, "*.cuh")) + \
        glob.glob(os.path.join(ROOT, "include", "*.h"))
    if not sources:
        raise RuntimeError("no CUDA sources under " + CSRC)
    obj_dir = OBJ + ("_bounds" if bounds else "")
    lib = LIB_BOUNDS if bounds else LIB
    os.makedirs(obj_dir, exist_ok=True)
    build_pycall(force)
    nvcc = _nvcc()
    extra = (["-Xptxas", "-v"] if verbose else []) + (["-DCKV_BOUNDS"] if bounds else [])
    hdr_time = _newest(headers) if headers else 0.0

    def compile_one(src: str) -> str:
        obj = os.path.join(obj_dir, os.path.basename(src)[:-3] + ".o")
        if force or not os.path.exists(obj) or os.path.getmtime(obj) < max(os.path.getmtime(src), hdr_time):
            cmd = [nvcc, *NVCC_FLAGS, *extra, "-c", src, "-o", obj]
            r = subprocess.run(cmd, capture_output=True, text=True)
            if verbose or r.returncode != 0:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed on " + src)
        return obj

    with concurrent.futures.ThreadPoolExecutor(max_workers=min(8, len(sources))) as ex:
        objs = list(ex.map(compile_one, sources))
    if force or not os.path.exists(lib) or os.path.getmtime(lib) < _newest(objs):
        tmp = lib + f".tmp{os.getpid()}"
        cmd = [nvcc, "-shared", "-o", tmp, *objs, "-Xlinker", "--exclude-libs,ALL"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv, bounds="--bounds" in sys.argv))
