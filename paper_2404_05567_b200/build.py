"""Builds ``libdsmoe.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a.

    python -m paper_2404_05567_b200.build [--force] [--verbose]

Each ``csrc/*.cu`` is compiled to an object under ``_build/`` (only when stale) and the objects are
linked into ``paper_2404_05567_b200/libdsmoe.so``.
"""
from __future__ import annotations

import concurrent.futures
import glob
import os
import subprocess
import sys

PKG = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(PKG)
CSRC = os.path.join(PKG, "csrc")
OBJ = os.path.join(ROOT, "_build")
LIB = os.path.join(PKG, "libdsmoe.so")

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC",
    "-I", os.path.join(ROOT, "include"), "-I", CSRC,
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def _stale(target: str, deps) -> bool:
    if not os.path.exists(target):
        return True
    t = os.path.getmtime(target)
    return any(os.path.getmtime(d) > t for d in deps)


def build(force: bool = False, verbose: bool = False) -> str:
    os.makedirs(OBJ, exist_ok=True)
    sources = sorted(glob.glob(os.path.join(CSRC, "*.cu")))
    headers = sorted(glob.glob(os.path.join(CSRC, "*.cuh"))) + [os.path.join(ROOT, "include", "dsmoe.h")]
    extra = ["-Xptxas", "-v"] if verbose else []
    extra += os.environ.get("DSMOE_NVCC_EXTRA", "").split()      # e.g. -DDSMOE_SMALL_INFLIGHT=196608 for a tuning build
    jobs = []
    objs = []
    for src in sources:
        obj = os.path.join(OBJ, os.path.basename(src)[:-3] + ".o")
        objs.append(obj)
        if force or _stale(obj, [src] + headers):
            jobs.append([_nvcc(), *NVCC_FLAGS, *extra, "-c", src, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with concurrent.futures.ThreadPoolExecutor(max_workers=8) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode != 0:
                sys.stderr.write(" ".join(cmd) + "\n" + r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed: " + cmd[-3])
    if jobs or force or _stale(LIB, objs):
        cmd = [_nvcc(), "-shared", "-o", LIB, *objs, "-Xcompiler", "-fPIC"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    return LIB


def build_variant(name: str, source: str, flags) -> str:
    """A second library for the tests: the built one with csrc/``source`` compiled with additional ``flags``."""
    build()
    lib, obj, src = (os.path.join(OBJ, f"libdsmoe_{name}.so"), os.path.join(OBJ, f"{name}.variant.o"), os.path.join(CSRC, source))
    others = [os.path.join(OBJ, os.path.basename(p)[:-3] + ".o") for p in sorted(glob.glob(os.path.join(CSRC, "*.cu"))) if p != src]
    if _stale(lib, [src, *others]):
        subprocess.run([_nvcc(), *NVCC_FLAGS, *flags, "-c", src, "-o", obj], check=True)
        subprocess.run([_nvcc(), "-shared", "-o", lib, obj, *others, "-Xcompiler", "-fPIC"], check=True)
    return lib


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="--verbose" in sys.argv))
