"""A CUDA call that fails is reported once, by the call that made it: the runtime's own record of the error, which plain
launches read back with cudaGetLastError(), is clear again afterwards.  The failing calls are stand-ins."""
import os
import subprocess

from paper_2104_08378_b200 import build

HARNESS = r"""
#include <cstdio>
#include "sp24_common.cuh"
using namespace sp24;
#ifndef __CUDA_ARCH__
static cudaError_t last = cudaSuccess;
static cudaError_t fail() { return last = cudaErrorInvalidConfiguration; }
extern "C" cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t*, const void*, void**) { return fail(); }
extern "C" cudaError_t cudaSetDevice(int) { return fail(); }
extern "C" cudaError_t cudaGetLastError() { cudaError_t e = last; last = cudaSuccess; return e; }
#endif
static void kernel(int) {}
static sp24_status checked() { SP24_CUDA_CHECK(cudaSetDevice(0)); return SP24_OK; }
int main() {
  const int launch = launch_overlapped(kernel, dim3(1), dim3(32), 0, nullptr, 1, 5);
  const int next = cuda_status(cudaGetLastError());
  const int call = checked();
  printf("%d %d %d %d", launch, next, call, (int)cuda_status(cudaGetLastError()));
}
"""


def failures(tmp_path, headers):
    """Status of a failed launch, of the plain launch after it, of another failed call, of the plain launch after that."""
    src, exe = tmp_path / "harness.cu", tmp_path / "harness"
    src.write_text(HARNESS)
    nvcc = build._nvcc()
    libs = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "shared", "-Xlinker",
                           f"-rpath={libs}", "-I", f"{build._ROOT}/include", "-I", headers, "-o", str(exe), str(src)])
    return subprocess.check_output([str(exe)], text=True).split()


def test_a_failed_call_leaves_no_error_behind(tmp_path):
    assert failures(tmp_path, f"{build._HERE}/csrc") == ["8", "0", "8", "0"]         # 8: SP24_ERR_CUDA
