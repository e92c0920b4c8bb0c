"""A launch that fails is reported once, by the call that made it: the runtime's own record of the error, which plain
launches read back with cudaGetLastError(), is clear again afterwards."""
import ctypes
import subprocess

from paper_2104_08378_b200 import build

HARNESS = r"""
#include "sp24_common.cuh"
using namespace sp24;
__global__ void nothing() {}
// A launch without blocks: refused on the host, with or without a device.
extern "C" int failed_launch() { return launch_overlapped(nothing, dim3(0), dim3(32), 0, nullptr, 1); }
static sp24_status checked() { SP24_CUDA_CHECK(cudaSetDevice(-1)); return SP24_OK; }
extern "C" int failed_call() { return checked(); }
extern "C" int last_error() { return (int)cudaPeekAtLastError(); }
"""


def test_a_failed_launch_leaves_no_error_behind(tmp_path):
    src, lib = tmp_path / "harness.cu", tmp_path / "harness.so"
    src.write_text(HARNESS)
    subprocess.check_call([build._nvcc(), *build.NVCC_FLAGS, "-I", f"{build._HERE}/csrc", "-o", str(lib), str(src)])
    h = ctypes.CDLL(str(lib))
    for failing in (h.failed_launch, h.failed_call):
        assert failing() == 8                # SP24_ERR_CUDA
        assert h.last_error() == 0
