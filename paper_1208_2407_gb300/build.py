"""Build libtrotter.so in-tree for sm_103a (nvcc, one -gencode, parallel TUs).

Usage: ``python -m paper_1208_2407_gb300.build [--force] [--verbose]``.
The library lands next to this file as ``libtrotter.so``; objects go to
``_build/`` at the repository root (git-ignored).
"""
from __future__ import annotations

import argparse
import concurrent.futures as cf
import os
import shutil
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
INCLUDE = os.path.join(ROOT, "include")
BUILD = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libtrotter.so")
SOURCES = ["api.cu", "tile.cu", "tile_adjoint.cu", "fused64.cu", "plain.cu", "reduce.cu", "adjoint.cu", "server.cu", "noalloc.cu",
           "lattice3d.cu", "selftest.cu"]
FUSED_PARTS = 16   # fused.cu is compiled in parts (-DTS_FUSED_PART=n), in parallel
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]


def nvcc() -> str:
    for cand in (os.environ.get("NVCC"), shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc"):
        if cand and os.path.exists(cand):
            return cand
    raise RuntimeError("nvcc not found (set NVCC or put CUDA's bin directory on PATH)")


def _flags(verbose: bool):
    f = ARCH + ["-O3", "-lineinfo", "-std=c++17", "-diag-suppress", "177", "-Xcompiler", "-fPIC", "-I" + INCLUDE,
                "-I" + CSRC]
    if verbose:
        f += ["-Xptxas", "-v"]
    return f


def _headers():
    return [os.path.join(CSRC, h) for h in os.listdir(CSRC) if h.endswith((".h", ".cuh"))] + \
        [os.path.join(INCLUDE, h) for h in os.listdir(INCLUDE) if h.endswith(".h")]


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    # (source, object, extra flags); fused.cu's parts first, they take longest
    units = [("fused.cu", "fused_%d.o" % n, ["-DTS_FUSED_PART=%d" % n])
             for n in reversed(range(FUSED_PARTS))]
    units += [(s, s.replace(".cu", ".o"), []) for s in SOURCES]
    newest_dep = max(os.path.getmtime(p) for p in _headers())
    objs, jobs = [], []
    for s, o, extra in units:
        src = os.path.join(CSRC, s)
        obj = os.path.join(BUILD, o)
        objs.append(obj)
        stale = (force or not os.path.exists(obj)
                 or os.path.getmtime(obj) < max(os.path.getmtime(src), newest_dep))
        if stale:
            jobs.append([nvcc(), "-c", src, "-o", obj] + extra + _flags(verbose))
    if jobs:
        with cf.ThreadPoolExecutor(max_workers=os.cpu_count() or 4) as ex:
            results = list(ex.map(lambda c: subprocess.run(c, capture_output=True, text=True), jobs))
        for cmd, r in zip(jobs, results):
            if verbose or r.returncode != 0:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if jobs or force or not os.path.exists(LIB) or \
            os.path.getmtime(LIB) < max(os.path.getmtime(o) for o in objs):
        tmp = LIB + ".%d.tmp" % os.getpid()
        cmd = [nvcc(), "-shared", "-o", tmp] + objs + ARCH + ["-Xcompiler", "-fPIC"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed: " + " ".join(cmd))
        os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    ap = argparse.ArgumentParser()
    ap.add_argument("--force", action="store_true")
    ap.add_argument("--verbose", action="store_true")
    a = ap.parse_args()
    print(build(force=a.force, verbose=a.verbose))
