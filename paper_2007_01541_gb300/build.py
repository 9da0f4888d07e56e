"""Build the solver's shared library (libwd.so) in-tree with nvcc for sm_103a.

Translation units are compiled in parallel; the library links the CUDA
runtime statically.  Output: paper_2007_01541_gb300/_build/libwd.so.
"""
from __future__ import annotations

import os
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(BUILD, "libwd.so")
SOURCES = ["csrc/symbolic.cpp", "csrc/api.cpp", "csrc/front_kernels.cu", "csrc/front64.cu", "csrc/solve_kernels.cu",
           "csrc/tc_schur.cu", "csrc/tc_chain.cu", "csrc/selinv.cu",
           "csrc/noalloc.cu", "csrc/batch.cu", "csrc/solve_blocked.cu", "csrc/tc_solve.cu",
           "csrc/lu.cu", "csrc/oz_schur.cu"]
HEADERS = ["csrc/symbolic.h", "csrc/engine.h", "csrc/dev_common.cuh", "csrc/tc_common.cuh",
           "csrc/front_block.cuh", "csrc/front64.cuh",
           "csrc/tile32.cuh"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def _nvcc() -> str:
    for c in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if c and (os.path.sep not in c or os.path.exists(c)):
            return c
    return "nvcc"


def _flags():
    return ARCH + ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O3",
                   "-I", os.path.join(ROOT, "include"), "--expt-relaxed-constexpr"]


def _stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    deps = [os.path.join(HERE, p) for p in SOURCES + HEADERS] + [os.path.join(ROOT, "include", "wd.h"),
                                                                 os.path.abspath(__file__)]
    return any(os.path.exists(p) and os.path.getmtime(p) > t for p in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    srcs = [s for s in SOURCES if os.path.exists(os.path.join(HERE, s))]
    if not force and not _stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    nvcc = _nvcc()

    def compile_one(src):
        obj = os.path.join(BUILD, os.path.basename(src) + ".o")
        cmd = [nvcc] + _flags() + ["-c", os.path.join(HERE, src), "-o", obj]
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed on {src}:\n{r.stdout}\n{r.stderr}")
        return obj

    with ThreadPoolExecutor(max_workers=len(srcs)) as ex:
        objs = list(ex.map(compile_one, srcs))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [nvcc] + ARCH + ["-shared", "-o", tmp] + objs + ["-lpthread", "-ldl", "-lrt"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
