"""Compile the CUDA library in-tree: csrc/*.cu -> libsp24.so (sm_100a SASS only), the sources side by side, and, beside a CUDA
build of torch, the binding's native part, csrc/sp24_native.cpp -> _native.<Python's ABI>.so.  The library needs nvcc only."""
from __future__ import annotations

import glob
import importlib.metadata
import importlib.util
import os
import subprocess
import sysconfig
import tempfile
from concurrent.futures import ThreadPoolExecutor

_HERE = os.path.dirname(os.path.abspath(__file__))
_ROOT = os.path.dirname(_HERE)
LIB_PATH = os.path.join(_HERE, "libsp24.so")
SOURCES = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cu")))
HEADERS = sorted(glob.glob(os.path.join(_HERE, "csrc", "*.cuh"))) + [os.path.join(_ROOT, "include", "sp24.h")]

NATIVE_PATH = os.path.join(_HERE, "_native" + sysconfig.get_config_var("EXT_SUFFIX"))
NATIVE_STAMP = os.path.join(_HERE, "_native.torch")     # the version of torch it was compiled against
NATIVE_SOURCES = [os.path.join(_HERE, "csrc", "sp24_native.cpp"), os.path.join(_ROOT, "include", "sp24.h")]

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


def _older(path: str, sources) -> bool:
    return not os.path.exists(path) or any(os.path.getmtime(f) > os.path.getmtime(path) for f in sources)


def _cuda_torch() -> tuple[str, str] | None:
    """Folder and version of the installed torch; None without one, or if it is a CPU-only build."""
    spec = importlib.util.find_spec("torch")
    if spec is None or spec.origin is None:
        return None
    folder = os.path.dirname(spec.origin)
    if not os.path.exists(os.path.join(folder, "lib", "libc10_cuda.so")):
        return None
    return folder, importlib.metadata.version("torch")


def _native_needs_build() -> bool:
    """Whether there is a native part to compile: missing, older than its sources, or for another torch."""
    torch = _cuda_torch()
    if torch is None:
        return False
    if _older(NATIVE_PATH, NATIVE_SOURCES) or not os.path.exists(NATIVE_STAMP):
        return True
    with open(NATIVE_STAMP) as f:
        return f.read() != torch[1]


def needs_build() -> bool:
    return _older(LIB_PATH, SOURCES + HEADERS) or _native_needs_build()


def _build_native() -> None:
    torch_dir, version = _cuda_torch()
    cuda_dir = os.path.dirname(os.path.dirname(_nvcc()))
    include = [os.path.join(_ROOT, "include"), os.path.join(torch_dir, "include"),
               os.path.join(torch_dir, "include", "torch", "csrc", "api", "include"), sysconfig.get_paths()["include"],
               os.path.join(cuda_dir or "/usr/local/cuda", "include")]
    tmp = f"{NATIVE_PATH}.{os.getpid()}.tmp"
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-fPIC", "-shared"] + [f"-I{d}" for d in include] +
                          ["-o", tmp, NATIVE_SOURCES[0], f"-L{torch_dir}/lib", "-lc10", "-lc10_cuda", "-ltorch_cpu", "-ltorch_python"])
    os.replace(tmp, NATIVE_PATH)
    with open(NATIVE_STAMP, "w") as f:
        f.write(version)


def build_library(force: bool = False, verbose: bool = False) -> str:
    """Compile what is missing or older than its sources (everything with force); returns the CUDA library's path."""
    if force or _older(LIB_PATH, SOURCES + HEADERS):
        tmp = f"{LIB_PATH}.{os.getpid()}.tmp"
        compile_ = [_nvcc()] + NVCC_FLAGS + (["-Xptxas", "-v"] if verbose else [])
        with tempfile.TemporaryDirectory() as objects, ThreadPoolExecutor(os.cpu_count()) as pool:
            names = [os.path.join(objects, os.path.basename(src) + ".o") for src in SOURCES]
            list(pool.map(lambda pair: subprocess.check_call(compile_ + ["-c", "-o", *pair]), zip(names, SOURCES)))
            subprocess.check_call([_nvcc()] + NVCC_FLAGS + ["--shared", "-o", tmp] + names)
        os.replace(tmp, LIB_PATH)
    if _native_needs_build() or (force and _cuda_torch() is not None):
        _build_native()
    return LIB_PATH


if __name__ == "__main__":
    print(build_library(force=True, verbose=True))
