"""Build ``liblbmhd.so`` (sm_103a) in-tree with nvcc.

The translation units under ``csrc/`` are compiled in parallel and linked
into one shared library next to this file; ``include/lbmhd.h`` is its C
ABI.  Nothing here needs a GPU.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import shutil
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "liblbmhd.so")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")

SOURCES = ["lbmhd_step.cu", "lbmhd_step_pipe.cu", "lbmhd_step_tma.cu", "lbmhd_aux.cu",
           "lbmhd_runtime.cu", "lbmhd_noalloc.cu", "lbmhd_batch.cu", "lbmhd_adjoint.cu",
           "lbmhd_kinetic.cu", "lbmhd3.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-std=c++17", "-lineinfo", "-Xcompiler", "-fPIC", "-Xcompiler", "-O2",
         "--expt-relaxed-constexpr", "-I", INCLUDE]
# Per-file flags.  The kinetic-LES kernels, the passes of several steps and the
# 3D step are compiled without FMA contraction: kernels of different shape
# (fused and two-pass; one or several steps; one or two nodes per thread)
# perform the same operations in the same order but in differently shaped
# code, and only with every fusion written out is "same operations" also
# "same bits".
FILE_FLAGS = {f: ["-fmad=false"] for f in ("lbmhd_step_pipe.cu", "lbmhd_kinetic.cu", "lbmhd3.cu")}


def nvcc() -> str:
    exe = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(exe):
        raise RuntimeError("nvcc not found")
    return exe


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "lbmhd.h"))
    files.append(os.path.abspath(__file__))
    return files


def stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(f) > t for f in _deps())


def build(force: bool = False, verbose: bool = False, extra_flags=()) -> str:
    """Compile and link; returns the library path.  Raises on failure."""
    if not force and not stale():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    cc = nvcc()

    def compile_one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        cmd = [cc, *ARCH, *FLAGS, *FILE_FLAGS.get(src, []), *extra_flags, "-c",
               os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stderr}")
        if verbose and r.stderr:
            print(r.stderr)
        return obj

    with cf.ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = LIB + f".{os.getpid()}.tmp"
    cmd = [cc, *ARCH, "-shared", "-o", tmp, *objs]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError("link failed:\n" + r.stderr)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    import sys

    print(build(force="--force" in sys.argv, verbose=True))
