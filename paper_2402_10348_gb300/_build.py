"""Builds libfsi.so (the CUDA library behind include/fsi.h) in-tree for sm_103a.

The translation units are compiled in parallel with nvcc and linked into
paper_2402_10348_gb300/libfsi.so.  Nothing else is built here.
"""
from __future__ import annotations

import os
import shutil
import subprocess
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OUT = os.path.join(HERE, "libfsi.so")
BUILD = os.path.join(HERE, "_build")
UNITS = ["api.cu", "ops_f64.cu", "ops_f32.cu", "krylov.cu", "step.cu", "gridcell.cu", "noalloc.cu", "pcnet.cu", "batch.cu", "diag.cu", "probe.cu", "tet.cu", "nsq_tma.cu", "nsa.cu", "hexq_ops.cu", "stencil.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "--expt-relaxed-constexpr"]
# the initialisation's integer results must not depend on FMA contraction
UNIT_FLAGS = {"gridcell.cu": ["-fmad=false"]}


def nvcc() -> str:
    for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libfsi")


def _stale() -> bool:
    if not os.path.exists(OUT):
        return True
    t = os.path.getmtime(OUT)
    srcs = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    srcs.append(os.path.join(HERE, "..", "include", "fsi.h"))
    return any(os.path.getmtime(s) > t for s in srcs if os.path.exists(s))


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return OUT
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()

    def one(u):
        obj = os.path.join(BUILD, u.replace(".cu", ".o"))
        extra = UNIT_FLAGS.get(u, [])
        cmd = [cc, *FLAGS, *extra, *ARCH, "-c", os.path.join(CSRC, u), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {u}:\n{r.stdout}\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    with ThreadPoolExecutor(max_workers=len(UNITS)) as ex:
        objs = list(ex.map(one, UNITS))
    tmp = OUT + ".tmp"
    cmd = [cc, "-shared", *ARCH, "-o", tmp, *objs, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force=True, verbose=True))
