"""Build the C-ABI library libamlbm.so in-tree with nvcc for sm_103a.

The translation units compile in parallel; the library lands next to this file
(paper_1310_1871_gb300/libamlbm.so) so that it is the one the binding loads.
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
INCLUDE = os.path.join(ROOT, "include")
OUT = os.path.join(HERE, "libamlbm.so")
BUILD = os.path.join(HERE, "_build")
SOURCES = ["amlbm_step.cu", "amlbm_step_pair.cu", "amlbm_step_split64.cu", "amlbm_step_strip.cu", "amlbm_step_row.cu",
           "amlbm_abi.cu", "amlbm_diag.cu", "amlbm_noalloc.cu", "amlbm_adjoint.cu", "amlbm_tune.cu", "amlbm_interface.cu"]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-O3", "-lineinfo", "-std=c++17", "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
# The step kernels state every fused multiply-add explicitly (rounding
# intrinsics); nothing else may be fused by the compiler, so that every
# schedule and tiling computes a site with the same operations.
FILE_FLAGS = {"amlbm_step.cu": ["-fmad=false"], "amlbm_step_pair.cu": ["-fmad=false"],
              "amlbm_step_split64.cu": ["-fmad=false"], "amlbm_step_strip.cu": ["-fmad=false"],
              "amlbm_step_row.cu": ["-fmad=false"]}


def _nvcc() -> str:
    for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if c and os.path.exists(c):
            return c
    raise RuntimeError("nvcc not found: the CUDA toolkit is required to build libamlbm.so")


def _stale() -> bool:
    if not os.path.exists(OUT):
        return True
    t = os.path.getmtime(OUT)
    deps = [os.path.join(CSRC, f) for f in os.listdir(CSRC)] + [os.path.join(INCLUDE, "amlbm.h")]
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    if not force and not _stale():
        return OUT
    nvcc = _nvcc()
    os.makedirs(BUILD, exist_ok=True)

    def compile_one(src):
        obj = os.path.join(BUILD, src.replace(".cu", ".o"))
        cmd = [nvcc, *ARCH, *FLAGS, *FILE_FLAGS.get(src, []), "-c", os.path.join(CSRC, src), "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
        return obj

    with cf.ThreadPoolExecutor(len(SOURCES)) as ex:
        objs = list(ex.map(compile_one, SOURCES))
    tmp = OUT + ".tmp"
    cmd = [nvcc, *ARCH, "-shared", "-o", tmp, *objs, "-lcudart"]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
    os.replace(tmp, OUT)
    return OUT


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True))
