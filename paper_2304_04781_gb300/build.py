"""Build libaewave.so (the C-ABI library) in-tree with nvcc for sm_103a.

Each translation unit is compiled in parallel, then linked into one shared library
next to this file.  Used by ``__graft_entry__.build()`` and by the binding when the
library is missing or older than its sources.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libaewave.so")
OBJ = os.path.join(HERE, "_build")
SOURCES = ["aew_api.cu", "aew_stencil.cu", "aew_reduce.cu", "aew_codec.cu", "aew_train.cu",
           "aew_revolve.cpp", "aew_pca.cpp", "aew_noalloc.cu", "aew_newton.cu", "aew_brick_fwd.cu",
           "aew_brick_incr.cu", "aew_brick_adj.cu", "aew_brick_cg.cu",
           "aew_twostep.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr"]


def nvcc() -> str:
    p = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(p):
        raise RuntimeError("nvcc not found; the CUDA toolkit is required to build aewave")
    return p


def _headers_mtime() -> float:
    t = 0.0
    for d in (CSRC, os.path.join(os.path.dirname(HERE), "include")):
        for f in os.listdir(d):
            if f.endswith((".h", ".cuh", ".cu", ".cpp")):
                t = max(t, os.path.getmtime(os.path.join(d, f)))
    return t


def up_to_date() -> bool:
    return os.path.exists(LIB) and os.path.getmtime(LIB) >= _headers_mtime()


def _compile(src: str, extra, objdir: str = OBJ) -> str:
    obj = os.path.join(objdir, os.path.splitext(src)[0] + ".o")
    cmd = [nvcc(), *ARCH, *FLAGS, *extra, "-c", os.path.join(CSRC, src), "-o", obj]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    return obj


def build(force: bool = False, verbose: bool = False, extra=(), out: str = LIB,
          objdir: str = OBJ) -> str:
    """Compile every source and link the library (default libaewave.so); returns its path."""
    if not force and out == LIB and up_to_date():
        return LIB
    os.makedirs(objdir, exist_ok=True)
    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(lambda s: _compile(s, list(extra), objdir), SOURCES))
    tmp = out + ".tmp"
    cmd = [nvcc(), *ARCH, "-shared", "-Xcompiler", "-fPIC", *objs, "-lpthread", "-o", tmp]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, out)
    if verbose:
        print(f"built {out}", file=sys.stderr)
    return out


if __name__ == "__main__":
    build(force="--force" in sys.argv, verbose=True)
