"""Builds libsclap.so (all CUDA sources, sm_103a) in place, with nvcc only.

Objects go to _build/ next to this file; sources compile in parallel and the
library is relinked only when a source or header is newer than it.  With
check=True (--check) it builds the bounds-check variant instead:
-DSCLAP_CHECK=1, objects in _build_check/, libsclap_check.so.
"""
from __future__ import annotations

import concurrent.futures as cf
import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
SO = os.path.join(HERE, "libsclap.so")
BUILD_CHECK = os.path.join(HERE, "_build_check")
SO_CHECK = os.path.join(HERE, "libsclap_check.so")
SOURCES = ["scan.cu", "lp.cu", "contract.cu", "ip.cu", "driver.cu", "noalloc.cu", "server.cu"]
HEADERS = [os.path.join(CSRC, "common.cuh"), os.path.join(CSRC, "arcs.cuh"), os.path.join(ROOT, "include", "sclap.h")]
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
FLAGS = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC"]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.sep not in cand or os.path.exists(cand)):
            return cand
    return "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False, check: bool = False) -> str:
    bdir, so = (BUILD_CHECK, SO_CHECK) if check else (BUILD, SO)
    flags = FLAGS + (["-DSCLAP_CHECK=1"] if check else [])
    os.makedirs(bdir, exist_ok=True)
    nvcc = _nvcc()
    jobs = []
    objs = []
    for src in SOURCES:
        s = os.path.join(CSRC, src)
        o = os.path.join(bdir, src.replace(".cu", ".o"))
        objs.append(o)
        if force or _stale(o, [s] + HEADERS):
            jobs.append([nvcc] + flags + ARCH + ["-c", s, "-o", o])

    def run(cmd):
        if verbose:
            print(" ".join(cmd), file=sys.stderr)
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            raise RuntimeError(f"nvcc failed:\n{' '.join(cmd)}\n{r.stdout}\n{r.stderr}")
        return cmd

    if jobs:
        with cf.ThreadPoolExecutor(max_workers=len(jobs)) as ex:
            list(ex.map(run, jobs))
    if force or jobs or _stale(so, objs):
        tmp = so + f".tmp{os.getpid()}"
        run([nvcc] + ARCH + ["-shared", "-o", tmp] + objs)
        os.replace(tmp, so)
    return so


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose=True, check="--check" in sys.argv))
