"""Build libtursca_gb.so in-tree with nvcc for sm_103a (GB300).

Each translation unit is compiled in parallel; the shared library links the
CUDA runtime dynamically.  Objects go to ``_build/`` beside this file and the
library to ``paper_2503_16037_gb300/libtursca_gb.so`` (both git-ignored).
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libtursca_gb.so")
INCLUDE = os.path.join(ROOT, "include")

SOURCES = ["graph.cpp", "persist_plan.cpp", "kernels_asm.cu", "kernels_solve.cu", "kernels_persist.cu", "kernels_render.cu", "kernels_adjoint.cu",
           "kernels_select.cu", "kernels_aniso.cu", "api.cu", "noalloc.cu", "selftest.cu", "server.cpp", "batch.cu"]
HEADERS = ["graph.h", "kern.h", "stage.cuh", "asm_util.cuh", "first_order.h", "select.h", "aniso.h", "aniso_mma.cuh", "aniso_contract.cuh", "batch.h", "persist.h", "persist_plan.h", "dots.cuh",
           "batcher.h"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found")
    return p


def _flags():
    return ARCH + ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC,-ffp-contract=off",
                   "-I", INCLUDE, "-I", CSRC]


def _stale(obj: str, src: str) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    deps = [src, os.path.join(INCLUDE, "tursca.h")] + [os.path.join(CSRC, h) for h in HEADERS]
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()
    jobs = []
    objs = []
    for s in SOURCES:
        src = os.path.join(CSRC, s)
        obj = os.path.join(BUILD, os.path.splitext(s)[0] + ".o")
        objs.append(obj)
        if force or _stale(obj, src):
            cmd = [cc] + _flags() + ["-c", src, "-o", obj]
            if s.endswith(".cpp"):
                cmd = [cc] + _flags() + ["-x", "c++", "-c", src, "-o", obj]
            jobs.append(cmd)
    with cf.ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 4))) as ex:
        futs = [ex.submit(subprocess.run, j, capture_output=True, text=True) for j in jobs]
        for j, f in zip(jobs, futs):
            r = f.result()
            if verbose or r.returncode != 0:
                sys.stderr.write(" ".join(j) + "\n" + r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed on %s" % j[-3])
    if jobs or not os.path.exists(LIB):
        tmp = LIB + ".%d.tmp" % os.getpid()
        cmd = [cc] + ARCH + ["-shared", "-cudart", "shared", "-o", tmp] + objs
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
