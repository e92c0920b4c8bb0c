// Shared host/device helpers of the sp24 library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "sp24.h"

namespace sp24 {

__host__ __device__ inline int elem_bytes(sp24_dtype t) {
  switch (t) {
    case SP24_F16:
    case SP24_BF16: return 2;
    case SP24_I8:
    case SP24_E4M3:
    case SP24_E5M2: return 1;
    case SP24_F32:
    case SP24_I32: return 4;
  }
  return 0;
}

inline bool is_fp8(sp24_dtype t) { return t == SP24_E4M3 || t == SP24_E5M2; }
// types of the 2:4 pattern (SP24_F32, the 1:2 pattern, is handled apart)
inline bool is_ab_type(sp24_dtype t) { return t == SP24_F16 || t == SP24_BF16 || t == SP24_I8 || is_fp8(t); }

inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// The current device must be a compute-capability 10.x part; the answer is cached per device.
sp24_status check_arch();

// SMs of the current device, cached per device (1 if there is none).
int sm_count();

// The status of a runtime call.  A call that fails also leaves its code behind as the thread's last error, which the
// plain launches read back with cudaGetLastError(): cleared here, so that only the call that failed reports it.
inline sp24_status cuda_status(cudaError_t e) {
  if (e == cudaSuccess) return SP24_OK;
  (void)cudaGetLastError();
  return SP24_ERR_CUDA;
}

// ---- launches that may start before the kernel ahead of them in the stream has ended -----------------
// A kernel launched through launch_overlapped() is set up (blocks scheduled as the ones of the kernel
// ahead leave their SMs, barriers and tables initialised) while that kernel drains; stream order is kept
// by wait_for_stream(), which every thread calls before its first access to global memory: it returns when
// all the work ahead has completed and its writes are visible.  Such a kernel takes no read-only
// (non-coherent) loads: its pointers carry no __restrict__ const, so that no load can be moved ahead of the wait.
// Blocks of the kernel behind may come in once every block of this one has ended or has called
// let_next_start(); it is a hint and orders nothing.  The GEMM calls it at its start, because its CTAs fill
// their SMs: the next one can only come to an SM that is idle.  The streaming kernels do not: with a call at
// the start, waiting blocks take the places of working ones (us a call in a CUDA graph, plain launches / called
// at the start / not called: prune_compress bf16 1184 x 1008 2.5, 3.3, 2.1; apply_mask i8 4096 x 768 3.9, 4.7, 3.7;
// apply_mask + compress bf16 1184 x 1008 4.4, 5.3, 4.0, of 12288 x 3072 44.8, 44.3, 44.1).
// Back-to-back calls (us a call, without and with the overlap): BERT FFN 17.7, 15.9; ragged 1184 x 736 x 1008
// 10.2, 8.3; int8 3072 x 4096 x 768 -> int8 19.9, 15.6; apply_mask + compress of 12288 x 3072 49.5, 44.7;
// in a CUDA graph 256 x 256 x 512 5.5, 4.6.
__device__ __forceinline__ void wait_for_stream() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void let_next_start() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <typename... Params, typename... Args>
inline sp24_status launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                     unsigned cluster, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  return cuda_status(cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...));
}

// ---- streaming kernels ----------------------------------------------------------------------------------
constexpr int kThreads = 256;

// A streaming kernel of few blocks behind a product: blocks that come in early find room only on the SMs that the product leaves
// idle, and all of them together there, where they then do the whole work.  So a launch of up to four blocks to an SM asks for as
// much (unused) shared memory as leaves room for an even spread only; the other blocks wait for the product's SMs.  Us a call in a
// CUDA graph, as they come and spread, each behind the product of its rows with 256 columns: prune_compress int8 3264 x 448 7.4,
// 6.1; bf16 3456 x 224 6.7, 5.5; 4448 x 448 8.2, 7.4; compress 7.0, 5.9; 6.3, 5.3; 7.9, 7.1; apply_mask and compress 8.2, 7.4; 7.5,
// 6.8; 10.2, 8.9.  By themselves, or behind other kernels, they take as long as before; without the early start 6.8, 6.2, 8.1.
template <auto KERNEL>
struct Kernel {};  // a kernel as an argument's type

template <auto KERNEL, typename... Args>
inline sp24_status launch_streaming(Kernel<KERNEL>, dim3 grid, dim3 block, cudaStream_t stream, Args... args) {
  static std::atomic<bool> allowed[64];  // the shared-memory opt-in, per kernel and device
  const int64_t sms = sm_count(), blocks_of_sm = sms > 0 ? ((int64_t)grid.x * grid.y + sms - 1) / sms : 0;
  constexpr int most = 227 * 1024 - 2048;  // (static shared memory and the KB that each block takes)
  int dev = 0;
  size_t smem = 0;
  if (blocks_of_sm >= 1 && blocks_of_sm <= 4 && cudaGetDevice(&dev) == cudaSuccess) {
    const bool kept = dev >= 0 && dev < 64;
    bool ok = kept && allowed[dev].load(std::memory_order_relaxed);
    if (!ok && (ok = cuda_status(cudaFuncSetAttribute(KERNEL, cudaFuncAttributeMaxDynamicSharedMemorySize, most)) == SP24_OK) && kept)
      allowed[dev].store(true, std::memory_order_relaxed);
    if (ok) smem = (size_t)(227 * 1024 / blocks_of_sm - 2048);
  }
  return launch_overlapped(KERNEL, grid, block, smem, stream, 1, args...);
}

__device__ __forceinline__ uint4 ld_stream(const void* p) { return __ldcs(reinterpret_cast<const uint4*>(p)); }
__device__ __forceinline__ void st_stream(void* p, uint4 v) { __stcs(reinterpret_cast<uint4*>(p), v); }
// 32 bytes at a 32-byte boundary, read or written once.
__device__ __forceinline__ void ld_stream32(const void* p, uint4 (&v)[2]) {
  asm volatile("ld.global.L1::no_allocate.L2::evict_first.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0].x), "=r"(v[0].y), "=r"(v[0].z), "=r"(v[0].w), "=r"(v[1].x), "=r"(v[1].y), "=r"(v[1].z), "=r"(v[1].w)
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st_stream32(void* p, const uint4 (&v)[2]) {
  asm volatile("st.global.L1::no_allocate.L2::evict_first.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(v[0].x),
               "r"(v[0].y), "r"(v[0].z), "r"(v[0].w), "r"(v[1].x), "r"(v[1].y), "r"(v[1].z), "r"(v[1].w)
               : "memory");
}

// What a kernel that works on cells (32 bytes of a row, see compress_kernel) may do with a whole one at once: read or write 32
// bytes, write 16 bytes of values of an 8-bit type.
enum { kWideX = 1, kWideY = 2, kWideVals = 4 };

// Block shape and grid of the vectorised kernels for `units` work units per row and `rows` rows:
// TX (a power of two, 32..256) threads along the row, chosen to waste the fewest lanes.
struct RowLaunch {
  dim3 grid, block;
  RowLaunch(int64_t units, int64_t rows, int unroll) {
    int best_tx = 256;
    int64_t best_cover = -1;
    for (int tx = 256; tx >= 32; tx /= 2) {
      int64_t per = (int64_t)tx * unroll;
      int64_t cover = (units + per - 1) / per * per;
      if (best_cover < 0 || cover < best_cover) { best_cover = cover; best_tx = tx; }
    }
    int ty = kThreads / best_tx;
    block = dim3((unsigned)best_tx, (unsigned)ty, 1);
    int64_t gy = (rows + ty - 1) / ty;
    if (gy > 32768) gy = 32768;
    grid = dim3((unsigned)(best_cover / ((int64_t)best_tx * unroll)), (unsigned)gy, 1);
  }
};

// The vectorised kernels hold offsets inside a row in 32 bits: of the matrix, and of the metadata in the operand order, where a
// row's bytes are spread over those of its 128-row block.  Longer rows are for the kernels of any alignment.
inline bool row_offsets_fit(int64_t K, int es, sp24_meta_layout l) {
  return (l == SP24_META_TCGEN05 ? (K + 255) / 256 * 4096 : K * es) <= int64_t(1) << 32;
}

#define SP24_RETURN_IF(cond, code) \
  do {                             \
    if (cond) return (code);       \
  } while (0)

#define SP24_CUDA_CHECK(expr)                                    \
  do {                                                           \
    if (cuda_status(expr) != SP24_OK) return SP24_ERR_CUDA;      \
  } while (0)

}  // namespace sp24
