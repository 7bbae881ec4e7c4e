"""Builds libbfc.so in-tree for sm_103a (nvcc, one -gencode, parallel units).

    python -m paper_1812_00283_gb300.build        # or build() from Python
"""
from __future__ import annotations

import concurrent.futures
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(PKG, "libbfc.so")
SOURCES = ["api.cu", "prepare.cu", "count.cu", "scan_sort.cu", "noalloc.cu", "server.cu", "microbench.cu",
           "derived.cu", "core.cu", "pairs.cu", "sparsify.cu"]
# (object, source, definitions): the count kernels are an object per mode and position type
UNITS = [(s[:-3] + ".o", s, []) for s in SOURCES]
UNITS += [(f"count_{mode}_{pos}.o", "count.cu", [f"-DBFC_COUNT_MODE={mode}", f"-DBFC_COUNT_POS={pos}"])
          for pos in ("int64_t", "int32_t") for mode in (4, 2, 1, 3, 0)]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libbfc")


def _flags(extra=()):
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE,
                   "-I", CSRC, "--expt-relaxed-constexpr", *extra]


def _stale(obj: str, src: str) -> bool:
    if not os.path.exists(obj):
        return True
    deps = [src, os.path.join(CSRC, "bfc_internal.cuh"), os.path.join(INCLUDE, "bfc.h")]
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, extra_flags=(), force: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    jobs = []
    for name, source, defs in reversed(UNITS):   # the long ones first
        src = os.path.join(CSRC, source)
        obj = os.path.join(BUILD, name)
        if force or _stale(obj, src):
            jobs.append([cc, *_flags(extra_flags), *defs, "-c", src, "-o", obj])
    if verbose:
        for j in jobs:
            print(" ".join(j))

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError("nvcc failed:\n" + " ".join(cmd) + "\n" + r.stdout + r.stderr)
        return r.stdout + r.stderr

    with concurrent.futures.ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        for out in ex.map(run, jobs):
            if verbose and out.strip():
                print(out)
    objs = [os.path.join(BUILD, name) for name, _, _ in UNITS]
    if force or jobs or not os.path.exists(LIB):
        tmp = LIB + f".tmp{os.getpid()}"
        run([cc, *ARCH, "-shared", "-cudart=static", "-Xlinker", "--no-undefined", "-o", tmp, *objs])
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
