"""The tile a product takes, the k-blocks of its stages, the CTAs that share a tile's k-blocks and the epilogue warps, as the
library's host code chooses them on a part with 148 SMs that holds as many clusters as a B200 was seen to (74 of 2 CTAs, 33 of
4, 15 of 8): sp24_gemm.cu compiled with stand-ins for the device queries and for the launch."""
import collections
import os
import subprocess

from paper_2104_08378_b200 import build

HARNESS = r"""
#include <cstdio>
#include <cstdlib>
#include "sp24_gemm.cuh"
#include "sp24_gemm_kernel.cuh"
namespace sp24 {
static int queries = 0;  // of the clusters that the device holds, since the last line
template <int KIND>
sp24_status report(TileShape t, bool sparse, bool b_mn, const sp24_gemm_desc* d, const GemmParams& p) {
  const int cs = elem_bytes(d->cd_type);
  auto kps = [&](auto c) {
    using C = decltype(c);
    return C::k_blocks_of_a_stage(t.tile_n, kEpiWarps * (C::staged_epilogue(cs, p.cd_col_major) ? 4096 : 2048), d->K / 2, p.conv != 0);
  };
  int k = 1;
  if (sparse && !b_mn && t.mblk == 1)
    k = t.ctas == 1 ? kps(Cfg<KIND, true, 128, 1, 1, false>{}) : t.block_n == 256 ? kps(Cfg<KIND, true, 256, 2, 1, false>{})
        : kps(Cfg<KIND, true, 224, 2, 1, false>{});
  const int warps = sparse && !b_mn && t.ctas == 2 && t.block_n == 224 && t.mblk == 1 ? epilogue_warps<KIND, true, 224, 2, 1, false>(d, t.tile_n) : kEpiWarps;
  printf("%dx%dx%d %d %d %d %d %d\n", t.ctas, t.block_n, t.mblk, t.tile_n, k, 1 << t.split_log, queries, warps);
  queries = 0;
  return SP24_OK;
}
#define SP24_KIND(K)                                                                                                          \
  template <> sp24_status launch_gemm<K>(TileShape t, bool s, bool b, const sp24_gemm_desc* d, const GemmParams& p, const void*, \
                                         const void*, const void*, cudaStream_t) { return report<K>(t, s, b, d, p); }
SP24_KIND(0) SP24_KIND(1) SP24_KIND(2) SP24_KIND(3)
sp24_status check_arch() { return SP24_OK; }
}
#include "sp24_gemm.cu"
#ifndef __CUDA_ARCH__
extern "C" cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
extern "C" cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr, int) { *v = 148; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) { return cudaSuccess; }
static int number(const char* name, int otherwise) { return getenv(name) ? atoi(getenv(name)) : otherwise; }
extern "C" cudaError_t cudaOccupancyMaxActiveClusters(int* n, const void*, const cudaLaunchConfig_t* cfg) {
  static int asked = 0;
  ++sp24::queries;
  if (asked++ < number("FAILING_QUERIES", 0)) return cudaErrorUnknown;
  *n = cfg->gridDim.x == 2 ? 74 : cfg->gridDim.x == 4 ? 33 : 15;
  if (number("NO_CLUSTERS", 0)) *n = 0;
  return cudaSuccess;
}
#endif
int main() {
  int ab, cd, dense, rows, cols, c;
  long long M, N, K;
  while (scanf("%d %d %lld %lld %lld %d %d %d %d", &ab, &cd, &M, &N, &K, &dense, &rows, &cols, &c) == 9) {
    sp24_gemm_desc d = {(sp24_dtype)ab, (sp24_dtype)cd, M, N, K, dense ? K : K / 2, rows ? N : K, cols ? M : N, cols ? M : N,
                        rows ? SP24_ROW_MAJOR : SP24_COL_MAJOR, cols ? SP24_COL_MAJOR : SP24_ROW_MAJOR,
                        cols ? SP24_COL_MAJOR : SP24_ROW_MAJOR, dense};
    const float f[2] = {1.f, c ? -1.5f : 0.f};
    const int32_t i[2] = {1, c};
    const bool whole = ab == SP24_I8;
    void* p = reinterpret_cast<void*>(16);
    const int st = whole && cd != SP24_I32 ? sp24_gemm_i8_dequant(&d, p, p, p, static_cast<float*>(p), nullptr, 0, 1.f, p, p, 256, nullptr) : sp24_gemm(&d, whole ? (const void*)i : f, p, p, p, whole ? (const void*)(i + 1) : f + 1, p, p, p, 256, nullptr);
    if (st != SP24_OK) printf("status %d\n", st);
  }
}
"""


def compile_harness(folder):
    """Path of the harness; choices(path, ...) below asks it."""
    src, exe = folder / "tile_choice.cu", folder / "tile_choice"
    src.write_text(HARNESS)
    nvcc = build._nvcc()
    libs = os.path.join(os.path.dirname(os.path.dirname(nvcc)), "lib64")
    subprocess.check_call([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-cudart", "shared", "-Xlinker",
                           f"-rpath={libs}", "-I", f"{build._ROOT}/include", "-I", f"{build._HERE}/csrc", "-o", str(exe), str(src)])
    return str(exe)


Choice = collections.namedtuple("Choice", "tile columns k_blocks parts queries warps")


def details(exe, problems, **env):
    """[Choice] for [(ab code, cd code, M, N, K, dense, N-contiguous B, column-major D, with C)], an int8 product with a result
    other than INT32 being the dequantised one.  FAILING_QUERIES=n: the device's answer to the first n questions for its
    clusters is an error; NO_CLUSTERS=1: it holds none."""
    text = "\n".join(" ".join(str(int(v)) for v in p) for p in problems)
    lines = subprocess.run([exe], input=text, capture_output=True, text=True, check=True,
                           env={**os.environ, **{name: str(value) for name, value in env.items()}}).stdout.splitlines()
    assert len(lines) == len(problems) and not any(line.startswith("status") for line in lines), lines
    return [Choice(tile, *map(int, rest)) for tile, *rest in (line.split() for line in lines)]


def choices(exe, problems):
    """[(tile, columns, k-blocks of a stage)] of details()."""
    return [(c.tile, c.columns, c.k_blocks) for c in details(exe, problems)]
