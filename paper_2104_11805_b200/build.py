"""Builds libsdnn.so (CUDA kernels + C ABI) in-tree for sm_100a with nvcc."""
from __future__ import annotations

import os
import subprocess
import sys

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "csrc")
LIB = os.path.join(HERE, "libsdnn.so")
SOURCES = [os.path.join(CSRC, "sdnn.cu")]
DEPENDS = SOURCES + [os.path.join(CSRC, "kernels.cuh"), os.path.join(CSRC, "vector.cuh"), os.path.join(CSRC, "resident.cuh"), os.path.join(CSRC, "resident.h"), os.path.join(CSRC, "plan.h"), os.path.join(CSRC, "capture.h"), os.path.join(CSRC, "reorder.h"), os.path.join(HERE, "..", "include", "sdnn.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-shared", "-Xcompiler", "-fPIC,-fopenmp,-O2", "-cudart", "static",
]


def up_to_date() -> bool:
    if not os.path.exists(LIB):
        return False
    t = os.path.getmtime(LIB)
    return all(os.path.getmtime(p) <= t for p in DEPENDS)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile the shared library next to this file; returns its path."""
    if not force and up_to_date():
        return LIB
    nvcc = os.environ.get("NVCC", "nvcc")
    cmd = [nvcc] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else []) + ["-o", LIB] + SOURCES + ["-lgomp", "-ldl"]
    subprocess.check_call(cmd)
    return LIB


if __name__ == "__main__":
    print(build_library(force="--force" in sys.argv, verbose="-v" in sys.argv))
