"""Build the in-tree CUDA library libkfbi.so for sm_103a with nvcc.

Each translation unit is compiled in parallel; setup.cu is compiled with
-fmad=false so that level sets, node coordinates and cell indices use
separately rounded multiplies and adds (bit-reproducible classification).
"""
from __future__ import annotations

import os
import shutil
import subprocess
import sys
from concurrent.futures import ThreadPoolExecutor

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
CSRC = os.path.join(HERE, "csrc")
BUILD = os.path.join(HERE, "_build")
LIB = os.path.join(HERE, "libkfbi.so")
INCLUDE = os.path.join(ROOT, "include")

# object: (source, extra flags); the transforms are compiled once per type, in parallel (each leaves the
# functions of the other type unused: warning 177)
OBJECTS = {
    "dst64.o": ("dst.cu", ["-DKFBI_DST_BITS=64", "-diag-suppress", "177"]),
    "dst32.o": ("dst.cu", ["-DKFBI_DST_BITS=32", "-diag-suppress", "177"]),
    "setup.o": ("setup.cu", ["-fmad=false"]),
    "ops.o": ("ops.cu", []),
    "capi.o": ("capi.cu", []),
    "noalloc.o": ("noalloc.cu", []),
    "mlp.o": ("mlp.cu", []),
}
ARCH = ["-gencode", "arch=compute_103a,code=sm_103a"]
COMMON = ["-std=c++17", "-O3", "-lineinfo", "-Xcompiler", "-fPIC", "-I" + INCLUDE, "-I" + CSRC]


def nvcc() -> str:
    path = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(path):
        raise RuntimeError("nvcc not found")
    return path


def _needs(obj: str, deps) -> bool:
    if not os.path.exists(obj):
        return True
    t = os.path.getmtime(obj)
    return any(os.path.getmtime(d) > t for d in deps)


def build(verbose: bool = False, force: bool = False) -> str:
    os.makedirs(BUILD, exist_ok=True)
    headers = [os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith(".cuh")]
    headers.append(os.path.join(INCLUDE, "kfbi.h"))
    jobs = []
    objs = []
    for name, (src, extra) in OBJECTS.items():
        path = os.path.join(CSRC, src)
        if not os.path.exists(path):
            continue
        obj = os.path.join(BUILD, name)
        objs.append(obj)
        if force or _needs(obj, [path] + headers):
            jobs.append([nvcc(), *COMMON, *ARCH, *extra, "-c", path, "-o", obj])

    def run(cmd):
        r = subprocess.run(cmd, capture_output=True, text=True)
        return cmd, r

    with ThreadPoolExecutor(max_workers=max(1, min(len(jobs), os.cpu_count() or 4))) as ex:
        for cmd, r in ex.map(run, jobs):
            if verbose or r.returncode != 0:
                sys.stderr.write(r.stdout + r.stderr)
            if r.returncode != 0:
                raise RuntimeError("nvcc failed: " + " ".join(cmd))
    if jobs or not os.path.exists(LIB) or _needs(LIB, objs):
        cmd = [nvcc(), "-shared", *ARCH, "-o", LIB, *objs, "-lcudart"]
        r = subprocess.run(cmd, capture_output=True, text=True)
        if r.returncode != 0:
            sys.stderr.write(r.stdout + r.stderr)
            raise RuntimeError("link failed")
    return LIB


if __name__ == "__main__":
    print(build(verbose="-v" in sys.argv, force="-f" in sys.argv))
