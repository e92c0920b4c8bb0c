// The GEMM kernels for FP16 and BF16 operands.
#include "sp24_gemm_kernel.cuh"

namespace sp24 {
template sp24_status launch_gemm<0>(TileShape, bool, bool, const sp24_gemm_desc*, const GemmParams&, const void*, const void*,
                                    const void*, cudaStream_t);
}  // namespace sp24
