// The GEMM kernels for 8-bit floating-point operands.
#include "sp24_gemm_kernel.cuh"

namespace sp24 {
template sp24_status launch_gemm<3>(TileShape, bool, bool, const sp24_gemm_desc*, const GemmParams&, const void*, const void*,
                                    const void*, cudaStream_t);
}  // namespace sp24
