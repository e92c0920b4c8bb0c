"""Compile the CUDA library in-tree: csrc/*.cu -> libsp24.so (sm_100a SASS only), the sources side by side."""
from __future__ import annotations

import glob
import os
import subprocess
import tempfile
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB_PATH = os.path.join(_HERE, "libsp24.so")
SOURCES = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))
HEADERS = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cuh"))) + [os.path.join(_ROOT, "include", "sp24.h")]

NVCC_FLAGS = [
    "-gencode", "arch=compute_100a,code=sm_100a", "-lineinfo", "-O3", "-std=c++17",
    "-Xcompiler", "-fPIC", "-cudart", "static",
    "-I", os.path.join(_ROOT, "include"),
]


def _nvcc() -> str:
    for cand in (os.environ.get("NVCC"), "/usr/local/cuda/bin/nvcc", "nvcc"):
        if cand and (os.path.isabs(cand) and os.path.exists(cand) or not os.path.isabs(cand)):
            return cand
    return "nvcc"


def needs_build() -> bool:
    if not os.path.exists(LIB_PATH):
        return True
    built = os.path.getmtime(LIB_PATH)
    return any(os.path.getmtime(f) > built for f in SOURCES + HEADERS)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Run nvcc if the library is missing or older than its sources; returns the .so path."""
    if force or needs_build():
        tmp = f"{LIB_PATH}.{os.getpid()}.tmp"
        compile_ = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else [])
        with tempfile.TemporaryDirectory() as objects, ThreadPoolExecutor(os.cpu_count()) as pool:
            names = [os.path.join(objects, os.path.basename(src) + ".o") for src in SOURCES]
            list(pool.map(lambda pair: subprocess.check_call(compile_ + ["-c", "-o", *pair]), zip(names, SOURCES)))
            subprocess.check_call([_nvcc()] + NVCC_FLAGS + ["--shared", "-o", tmp] + names)
        os.replace(tmp, LIB_PATH)
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
