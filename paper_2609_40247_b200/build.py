"""Builds the CUDA library (libta.so) for sm_100a with nvcc and the tensor helpers of the Python
binding (_views.so) with g++, in-tree.

    python -m paper_2609_40247_b200.build [--force] [--verbose]
"""
from __future__ import annotations

import glob
import os
import subprocess
import sys
import sysconfig
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
OBJ = os.path.join(HERE, "build")
LIB = os.path.join(HERE, "libta.so")
NVCC = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
         "-Xcompiler", "-fPIC"] + os.environ.get("TA_DEFS", "").split()


VIEWS_SRC = os.path.join(CSRC, "views.cpp")
VIEWS = os.path.join(HERE, "_views.so")


def build_views(force: bool = False) -> str:
    """The tensor helpers of the Python binding (g++, against the installed torch)."""
    if not force and os.path.exists(VIEWS) and os.path.getmtime(VIEWS) >= os.path.getmtime(VIEWS_SRC):
        return VIEWS
    import torch
    base = os.path.dirname(torch.__file__)
    inc = [os.path.join(base, "include"), os.path.join(base, "include", "torch", "csrc", "api", "include"),
           sysconfig.get_paths()["include"], os.path.join(os.path.dirname(os.path.dirname(NVCC)), "include")]
    cmd = ["g++", "-O2", "-std=c++17", "-shared", "-fPIC", f"-D_GLIBCXX_USE_CXX11_ABI={int(torch._C._GLIBCXX_USE_CXX11_ABI)}",
           VIEWS_SRC, "-o", VIEWS + ".tmp", "-L" + os.path.join(base, "lib"), "-ltorch_python", "-ltorch_cpu", "-lc10"]
    r = subprocess.run(cmd + ["-I" + i for i in inc], capture_output=True, text=True)
    if r.returncode != 0:
        raise RuntimeError(f"g++ failed for {VIEWS_SRC}:\n{r.stdout}\n{r.stderr}")
    os.replace(VIEWS + ".tmp", VIEWS)
    return VIEWS


def sources():
    return sorted(glob.glob(os.path.join(CSRC, "*.cu")))


def _deps_mtime():
    hs = glob.glob(os.path.join(CSRC, "*.cuh")) + [os.path.join(HERE, "..", "include", "ta.h")]
    return max(os.path.getmtime(h) for h in hs)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    dep = _deps_mtime()
    jobs = []
    objs = []
    for src in sources():
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        stale = (not os.path.exists(obj)) or os.path.getmtime(obj) < max(os.path.getmtime(src), dep)
        if force or stale:
            jobs.append((src, obj))

    def compile_one(job):
        src, obj = job
        cmd = [NVCC] + FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-c", src, "-o", obj]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed for {src}:\n{r.stdout}\n{r.stderr}")
        if verbose:
            sys.stderr.write(r.stderr)
    with ThreadPoolExecutor(max_workers=8) as ex:
        views = ex.submit(build_views, force)
        list(ex.map(compile_one, jobs))
        views.result()
    if jobs or not os.path.exists(LIB):
        # drop objects of sources that no longer exist
        for o in glob.glob(os.path.join(OBJ, "*.o")):
            if o not in objs:
                os.remove(o)
        cmd = [NVCC, "-shared", "-o", LIB + ".tmp"] + objs + ["-gencode", "arch=compute_100a,code=sm_100a"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"link failed:\n{r.stdout}\n{r.stderr}")
        os.replace(LIB + ".tmp", LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
