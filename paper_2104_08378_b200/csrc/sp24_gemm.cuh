// What the host side of the GEMM (sp24_gemm.cu) and its kernels (sp24_gemm_kernel.cuh) share.
#pragma once

#include <cuda.h>

#include "sp24_common.cuh"

namespace sp24 {

constexpr int kBlockM = 128;              // rows of A per CTA and m-block (tensor-memory lanes)
constexpr int kAtomBytes = 128;           // bytes per row of one swizzle-128B operand atom
constexpr int kEpiWarps = 8;              // two per tensor-memory lane quarter, taking alternate boxes
constexpr int kFirstEpiWarp = 2;          // warp 0: TMA producer, warp 1: MMA issuer
constexpr int kNumThreads = 32 * (kFirstEpiWarp + kEpiWarps);
// (Ten warps leave three on two of the SM's four sub-partitions, which caps the kernel at 168
// registers per thread; trading registers between the roles with setmaxnreg was tried and made the
// compiler spill far more than it saved.)
constexpr long long kWaitTimeoutCycles = 2000ll * 1000ll * 1000ll;  // per wait: 1-2 s of SM clock
constexpr uint32_t kTmemCols = 512;

// n / d for n < 2^31 by a multiplication (Granlund and Montgomery, Division by Invariant Integers using Multiplication): mul / 2^(31 + log) is 1 / d rounded up, by less than 2^-31 / d, with 2^log the
// first power of two >= d.  (A division by a divisor known only at run time takes the device about 150 cycles, and the
// first load of a call waits for two.)
struct FastDiv {
  uint32_t mul, shift;
  static FastDiv by(uint32_t d) {
    uint32_t log = 0;
    while ((uint64_t(1) << log) < d) ++log;
    return {(uint32_t)((uint64_t(1) << (31 + log)) / d + 1), 31 + log};
  }
  __host__ __device__ __forceinline__ int operator()(int n) const { return (int)(((uint64_t)(uint32_t)n * mul) >> shift); }
};

// The owner of a ring of barriers waits, after its last use of them, once for every slot, in the order in which it would use
// them next and for what it would wait for then: `slot` and `phase` are those of its next use, wait(slot, parity) is its
// wait for a free slot (at once for one that was never used).  After that nothing is on its way to these barriers.
template <class Wait>
__host__ __device__ __forceinline__ bool drain_ring(int slots, int slot, uint32_t phase, Wait wait) {
  for (int i = 0; i < slots; ++i) {
    if (!wait(slot, phase ^ 1u)) return false;
    if (++slot == slots) { slot = 0; phase ^= 1u; }
  }
  return true;
}

struct GemmParams {
  int64_t M, N, K;
  int64_t ldc, ldd;   // elements
  const void* C;
  void* D;
  uint32_t* status;   // [0] = 0 ok, else code of the first wait that expired; [1] = number of expired waits
  float alpha, beta;
  int32_t m_tiles, n_tiles, k_blocks;
  int32_t meta_kb;    // 128-column metadata blocks per 128-row block (K padded to 256)
  int32_t a_fmt;      // 0 f16, 1 bf16 (kind::f16); ignored for int8
  int32_t cd_type;    // sp24_dtype of C / D
  int32_t has_c;
  int32_t stages, epi_bytes;  // shared memory: ring stages and bytes of epilogue staging
  long long wait_limit;       // SM cycles after which a device-side wait gives up
  int32_t test_skip_stage;    // test hook: the producers leave out one k-block, so that a wait expires (2 + r: only CTA r of those that share a tile's)
  int32_t band;       // m-tiles per band of the tile sweep
  FastDiv by_band_tiles, by_band, by_last_band;  // tiles of a band; m-tiles of a band and of the last one
  int32_t tile_n;     // columns of a tile: the kernel's BLOCK_N or fewer
  int32_t kps;        // k-blocks of a stage (1 or 2)
  int32_t split_log;  // log2 of the CTAs (a cluster) that share a tile's k-blocks; INT32 accumulators of single CTAs only
  int32_t part_bytes; // ... and the room for the other CTAs' parts of the boxes that a CTA finishes
  int32_t mblk, b_stages;  // tall tiles only: m-blocks of a tile, slots of the B ring
  int32_t b_3d;       // map_b is three-dimensional: a stage of B is one load
  int32_t cd_col_major;  // C and D stored M-contiguous (the [tokens, out_features] layout): selects the kernel
  // implicit 3x3 convolution: B is the im2col view of an NHWC activation (never materialised)
  int32_t conv, conv_h, conv_w, conv_c;
  FastDiv by_image, by_conv_w;  // pixels of an image, of an image row
  // int8 dequantising epilogue (sp24_gemm_i8_dequant): out = act(row_scale[i] * acc + bias[i]),
  // requantised with out_inv_scale when the output type is int8
  int32_t dequant, relu;
  int32_t acc_f16;    // FP16 accumulation (kind::f16 with a binary16 accumulator; FP16 operands only)
  const float* row_scale;
  const float* bias;
  float out_inv_scale;
};

constexpr int kSwizzle128Atom32 = 1280;

// Up to three dimensions, innermost first: sizes in elements, strides of the outer ones in bytes.
struct MapShape {
  const void* base;
  uint64_t dims[3], strides[2];  // dims[2] == 0: two dimensions
  uint32_t box[3];
  int32_t es, swizzle;  // swizzle: 0, 128, or kSwizzle128Atom32 = the 128-byte pattern in 32-byte units
  bool operator==(const MapShape& o) const {
    return base == o.base && dims[0] == o.dims[0] && dims[1] == o.dims[1] && dims[2] == o.dims[2] &&
           strides[0] == o.strides[0] && strides[1] == o.strides[1] && box[0] == o.box[0] && box[1] == o.box[1] &&
           box[2] == o.box[2] && es == o.es && swizzle == o.swizzle;
  }
};

// ---- in sp24_gemm.cu -----------------------------------------------------------------------------
sp24_status make_map(CUtensorMap* map, const MapShape& key);  // from a small cache, or encoded
// 2-D map over a row-major (rows x cols) array of `es`-byte elements with `ld_bytes` between rows; box = box_cols x
// box_rows elements.
inline sp24_status make_map(CUtensorMap* map, const void* base, int es, uint64_t rows, uint64_t cols, uint64_t ld_bytes,
                            uint32_t box_cols, uint32_t box_rows, int swizzle) {
  return make_map(map, MapShape{base, {cols, rows, 0}, {ld_bytes, 0}, {box_cols, box_rows, 1}, es, swizzle});
}
sp24_status make_im2col_map(CUtensorMap* map, const void* x, int es, uint64_t nb, uint64_t h, uint64_t w, uint64_t c,
                            uint32_t channels_per_box, uint32_t pixels_per_box);

// ---- in sp24_gemm_{f16,i8,tf32,f8}.cu --------------------------------------------------------------
// One launch of the kernel for MMA kind KIND (0 = f16 / bf16, 1 = int8, 2 = tf32, 3 = 8-bit floating point (e4m3 /
// e5m2)) with tiles of ctas x block_n x mblk of which tile_n columns are used; SP24_ERR_UNSUPPORTED if that shape is not
// built.  Each kind is instantiated in a source file of its own, so that they compile side by side.
struct TileShape {
  int ctas, block_n, mblk, tile_n;
  int split_log;  // see GemmParams
};
template <int KIND>
sp24_status launch_gemm(TileShape tile, bool sparse, bool b_mn, const sp24_gemm_desc* d, const GemmParams& p, const void* A,
                        const void* meta, const void* B, cudaStream_t s);

}  // namespace sp24
