"""Builds the CUDA library (sm_100a only) in-tree, paper_2609_33503_b200/librelaxkv.so, and the Python module through which the
binding calls it, paper_2609_33503_b200/_calls.so.

nvcc cross-compiles without a GPU.  Each .cu file is one translation unit, compiled in parallel.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys
import sysconfig

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
INCLUDE = os.path.join(os.path.dirname(HERE), "include")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "librelaxkv.so")
CALLS = os.path.join(HERE, "_calls.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC", "-I", INCLUDE, "-I", CSRC]
# RELAXKV_NVTX=1: compile NVTX ranges into every C-ABI call and kernel launch (the header-only NVTX v3 of the toolkit);
# objects of the two flavours are kept apart
NVTX = os.environ.get("RELAXKV_NVTX", "0") not in ("", "0")
if NVTX:
    FLAGS += ["-DRELAXKV_NVTX"]
    OBJ = os.path.join(HERE, "build_nvtx")


def sources():
    return sorted(f for f in os.listdir(CSRC) if f.endswith(".cu"))


def _newest_header() -> float:
    hs = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    hs += [os.path.join(INCLUDE, f) for f in os.listdir(INCLUDE)]
    return max(os.path.getmtime(h) for h in hs)


def build(force: bool = False, verbose: bool = False, ptxas_v: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    hdr = _newest_header()
    jobs = []
    for src in sources():
        s = os.path.join(CSRC, src)
        o = os.path.join(OBJ, src[:-3] + ".o")
        if force or not os.path.exists(o) or os.path.getmtime(o) < max(os.path.getmtime(s), hdr):
            cmd = [NVCC, *FLAGS, "-c", s, "-o", o]
            if ptxas_v:
                cmd[1:1] = ["-Xptxas", "-v"]
            jobs.append((src, cmd))
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=min(8, len(jobs))) as ex:
            futs = {ex.submit(subprocess.run, cmd, capture_output=True, text=True): src for src, cmd in jobs}
            for f in cf.as_completed(futs):
                r = f.result()
                if verbose or ptxas_v or r.returncode != 0:
                    sys.stderr.write(f"--- {futs[f]} ---\n{r.stdout}{r.stderr}\n")
                if r.returncode != 0:
                    raise RuntimeError(f"nvcc failed on {futs[f]}")
    objs = [os.path.join(OBJ, s[:-3] + ".o") for s in sources()]
    if jobs or not os.path.exists(LIB) or any(os.path.getmtime(o) > os.path.getmtime(LIB) for o in objs):
        tmp = LIB + f".tmp{os.getpid()}"
        subprocess.check_call([NVCC, "-shared", "-o", tmp, *objs, *(["-ldl"] if NVTX else [])])
        os.replace(tmp, LIB)
    build_calls(force)
    return LIB


def build_calls(force: bool = False) -> str:
    src, header = os.path.join(CSRC, "py_calls.cpp"), os.path.join(INCLUDE, "relaxkv.h")
    if force or not os.path.exists(CALLS) or os.path.getmtime(CALLS) < max(os.path.getmtime(src), os.path.getmtime(header)):
        tmp = CALLS + f".tmp{os.getpid()}"
        subprocess.check_call([os.environ.get("CXX", "g++"), "-shared", "-fPIC", "-O2", "-std=c++17", "-Wall", "-I", INCLUDE,
                               "-I", sysconfig.get_paths()["include"], src, "-o", tmp])
        os.replace(tmp, CALLS)
    return CALLS


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, ptxas_v="--ptxas" in sys.argv))
