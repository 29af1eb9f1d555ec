"""Builds ``libpacer.so`` (the C-ABI CUDA library) in-tree with nvcc for sm_100a."""
from __future__ import annotations

import os
import subprocess
import sys
import tempfile
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(_HERE, "csrc")
LIB = os.path.join(_HERE, "libpacer.so")

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-Xcompiler", "-fPIC", "--use_fast_math=false"]


def _sources():
    return sorted(os.path.join(CSRC, f) for f in os.listdir(CSRC) if f.endswith((".cu", ".cuh", ".h"))) + \
        [os.path.join(os.path.dirname(_HERE), "include", "pacer.h")]


def needs_build() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(s) > t for s in _sources())


def build_lib(force: bool = False, verbose: bool = False) -> str:
    """Compile csrc/*.cu into libpacer.so if it is missing or older than a source."""
    if not force and not needs_build():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    cus = [s for s in _sources() if s.endswith(".cu")]
    tmp = LIB + ".tmp.%d" % os.getpid()
    flags = [f for f in NVCC_FLAGS if not f.startswith("--use_fast_math")]
    with tempfile.TemporaryDirectory() as d:                # one process per translation unit
        objs = [os.path.join(d, os.path.basename(c) + ".o") for c in cus]
        extra = ["-Xptxas", "-v"] if verbose else []
        with ThreadPoolExecutor(max_workers=os.cpu_count() or 1) as pool:
            list(pool.map(lambda co: subprocess.check_call([nvcc] + flags + extra + ["-c", "-o", co[1], co[0]]), zip(cus, objs)))
        subprocess.check_call([nvcc] + flags + ["-shared", "-o", tmp] + objs)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build_lib(force="--force" in sys.argv, verbose="-v" in sys.argv))
