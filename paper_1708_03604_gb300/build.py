"""Build libbsm.so (the C-ABI library) in-tree with nvcc for sm_103a.

Each CUDA translation unit is compiled in parallel into ``_build/`` next to
this file, then linked into ``libbsm.so`` in the package directory.  A unit
is recompiled only when it or a header is newer than its object file.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libbsm.so")
# the debug build: device-side bounds checks in the numeric kernels (-DBSM_DEBUG)
BUILD_DEBUG = os.path.join(PKG, "_build_debug")
LIB_DEBUG = os.path.join(PKG, "libbsm_debug.so")
SOURCES = ["bsm_api.cu", "k_symbolic.cu", "k_numeric.cu", "k_split_tf32x3.cu", "k_split_bf16x3.cu",
           "k_split_bf16x6.cu", "k_group.cu", "k_tile.cu", "k_warp.cu", "k_add.cu", "k_panel.cu",
           "bsm_static.cu", "k_probe.cu"]
HEADERS = [os.path.join(CSRC, "bsm_internal.cuh"), os.path.join(CSRC, "numeric_debug.cuh"),
           os.path.join(CSRC, "numeric_split.cuh"), os.path.join(CSRC, "numeric_warp.cuh"),
           os.path.join(CSRC, "numeric_items.cuh"), os.path.join(ROOT, "include", "bsm.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "-I" + os.path.join(ROOT, "include")]


def nvcc() -> str:
    cand = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return cand if os.path.exists(cand) else "nvcc"


def _stale(obj: str, src: str) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(p) > t for p in [src] + HEADERS)


def build(verbose: bool = False, force: bool = False, debug: bool = False) -> str:
    """Compile libbsm.so (debug=True: libbsm_debug.so with -DBSM_DEBUG)."""
    bdir, lib = (BUILD_DEBUG, LIB_DEBUG) if debug else (BUILD, LIB)
    flags = FLAGS + (["-DBSM_DEBUG=1"] if debug else [])
    os.makedirs(bdir, exist_ok=True)
    jobs = []
    objs = []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(bdir, s.replace(".cu", ".o"))
        objs.append(obj)
        if force or _stale(obj, src):
            jobs.append([nvcc(), *ARCH, *flags, "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        if verbose and (r.stdout or r.stderr):
            sys.stderr.write(r.stdout + r.stderr)

    with ThreadPoolExecutor(max_workers=max(1, len(jobs))) as ex:
        list(ex.map(run, jobs))
    if jobs or not os.path.exists(lib) or any(os.path.getmtime(o) > os.path.getmtime(lib) for o in objs):
        tmp = lib + f".tmp{os.getpid()}"
        run([nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"])
        os.replace(tmp, lib)
    return lib


if __name__ == "__main__":
    print(build(verbose=True, force="--force" in sys.argv, debug="--debug" in sys.argv))
