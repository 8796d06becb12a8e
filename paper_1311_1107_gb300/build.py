"""Build libqedpic.so in-tree with nvcc for sm_103a.

Each translation unit is compiled in parallel to an object file, then the
objects are linked into ``paper_1311_1107_gb300/_build/libqedpic.so``.
Usage: ``python -m paper_1311_1107_gb300.build [--force]``.
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(PKG, "_build")
LIB = os.path.join(BUILD, "libqedpic.so")

SOURCES = ["qp_step_fp64.cu", "qp_step_mixed.cu", "qp_kernels.cu", "qp_abi.cu", "qp_noalloc.cu",
           "qp_coalesce.cu", "qp_pic.cu", "qp_tables.cpp"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
# Per-unit flags.  The mixed-precision step divides in FP32 with the
# hardware reciprocal (2 ulp): its tolerance is set by FP32 physics, and the
# IEEE division's range checks and slow path cost more than the division.
# The FP64 step keeps IEEE division and square root where it calls them; most of
# its quotients and roots are Newton iterations within a unit of the last place.
# The coalescence forms its groups and sums with the oracle's FP64
# operations in the oracle's order: no FMA contraction there.
UNIT_FLAGS = {"qp_step_mixed.cu": ["-prec-div=false"], "qp_coalesce.cu": ["-fmad=false"]}


def nvcc() -> str:
    cand = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(cand):
        raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libqedpic")
    return cand


def _deps():
    files = [os.path.join(CSRC, f) for f in os.listdir(CSRC)]
    files.append(os.path.join(INCLUDE, "qedpic.h"))
    files.append(os.path.abspath(__file__))
    return files


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(f) <= t for f in _deps())


def _compile(src: str, verbose: bool) -> str:
    obj = os.path.join(BUILD, os.path.splitext(src)[0] + ".o")
    cmd = [nvcc(), *ARCH, "-lineinfo", "-O3", "-std=c++17", "-Xcompiler", "-fPIC,-O2",
           *UNIT_FLAGS.get(src, []), "-I", INCLUDE, "-I", CSRC, "-c", os.path.join(CSRC, src),
           "-o", obj]
    if src.endswith(".cu"):
        cmd[5:5] = ["-Xptxas", "-v"] if verbose else []
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
    if verbose and (r.stdout or r.stderr):
        sys.stderr.write(r.stdout + r.stderr)
    return obj


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and up_to_date():
        return LIB
    os.makedirs(BUILD, exist_ok=True)
    with ThreadPoolExecutor(max_workers=len(SOURCES)) as ex:
        objs = list(ex.map(lambda s: _compile(s, verbose), SOURCES))
    tmp = LIB + f".tmp{os.getpid()}"
    cmd = [nvcc(), *ARCH, "-shared", "-o", tmp, *objs, "-lpthread"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
