"""Build the CUDA library in-tree for sm_100a (nvcc cross-compiles without a GPU)."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsailor_b200.so")
SOURCES = [os.path.join(CSRC, f) for f in ("sailor_lib.cu", "sailor_plan_obj0.cu", "sailor_plan_obj1.cu", "sailor_plan_obj2.cu")]
DEPS = SOURCES + [os.path.join(CSRC, f) for f in ("sailor_tables.cuh", "sailor_plan_kernels.cuh", "sailor_plan_setup.cuh", "sailor_dp.cuh", "sailor_dp_budget.cuh", "sailor_batch.cuh", "sailor_mixed.cuh", "sailor_mixed_batch.cuh", "sailor_mixed_search.cuh", "sailor_peaks.cuh")] + [
    os.path.join(os.path.dirname(HERE), "include", "sailor.h")]

NVCC_FLAGS = ["-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
              "-fmad=false", "--compress-mode=size", "-shared", "-Xcompiler", "-fPIC"]


def is_stale() -> bool:
    if not os.path.exists(LIB):
        return True
    t = os.path.getmtime(LIB)
    return any(os.path.getmtime(d) > t for d in DEPS)


def build(force: bool = False, verbose: bool = False) -> str:
    """Compile libsailor_b200.so next to this file; returns its path."""
    if not force and not is_stale():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    tmp = LIB + f".{os.getpid()}.tmp"
    objects = [f"{tmp}.{j}.o" for j in range(len(SOURCES))]
    flags = [f for f in NVCC_FLAGS if f != "-shared"] + (["-Xptxas", "-v"] if verbose else [])
    running = [subprocess.Popen([nvcc] + flags + ["-c", "-o", obj, src]) for src, obj in zip(SOURCES, objects)]   # side by side
    try:
        failed = [p.args for p in running if p.wait() != 0]
        if failed:
            raise subprocess.CalledProcessError(1, failed[0])
        subprocess.check_call([nvcc] + NVCC_FLAGS + ["-o", tmp] + objects)
    finally:
        for obj in objects:
            if os.path.exists(obj):
                os.remove(obj)
    os.replace(tmp, LIB)
    return LIB


if __name__ == "__main__":
    print(build(force="--force" in sys.argv, verbose="-v" in sys.argv))
