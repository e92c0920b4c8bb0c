// D = alpha * A * B + beta * C on the sm_100a tensor cores (Section 3.2, Figure 2 of arXiv
// 2104.08378): A is either 2:4-compressed (values + metadata, tcgen05.mma.sp) or dense
// (tcgen05.mma, the "dense variant" that supplies the sparse-vs-dense speedup).
//
// One persistent, warp-specialised kernel:
//   warp 0   TMA producer: compressed-A tiles, metadata blocks and B tiles of one k-block into a
//            ring of shared-memory stages (mbarrier expect_tx / complete_tx);
//   warp 1   MMA issuer (one elected thread): copies the stage's metadata shared -> tensor
//            memory (tcgen05.cp), issues the tcgen05.mma[.sp] of the stage, commits the stage
//            back to the producer and, after the last k-block, the accumulators to the epilogue;
//            owns the tensor-memory allocation;
//   warps 2-9 epilogue (2-13 in the kernels of twelve_warps), two (three) per tensor-memory lane quarter taking 32-column boxes
//            in turn:
//            tcgen05.ld accumulator -> registers, alpha / beta / conversion in registers, then one of two
//            forms.  4-byte row-major outputs: a
//            staging box per warp, C boxes TMA-loaded one box ahead, TMA store of the D box, if
//            shared memory has room for the boxes.  All others: the warps load C and store D
//            themselves, through a small transposing buffer per warp, and hand the accumulators back
//            as soon as their last box is in registers.
// CTAS == 2 runs a pair of CTAs (cluster of two): each CTA loads its 128 rows of A / metadata per
// m-block and its half of B, CTA 0 issues cta_group::2 MMAs (M = 256) for both.
// SPLIT runs a cluster of 2, 4 or 8 CTAs on one tile of INT32 sums, each with a part of the k-blocks
// and MMAs of its own; the epilogue warps exchange the accumulators.
// MBLK == 2 gives every CTA two m-blocks (two accumulators, one B tile): what an SM can pull in
// from the L2 per clock, not the tensor pipe, bounds this kernel, and sharing the B tile between
// two m-blocks cuts the bytes per flop by about a third.  The two accumulators then fill tensor
// memory, so the epilogue is not overlapped with the next tile's main loop; MBLK == 1 keeps two
// accumulator buffers and overlaps it.
// Every wait is bounded: on expiry the role records a code in the status record and all roles
// leave through the normal teardown (no trap, no endless spin).  The kernel never clears the
// record: it stays at the first expired wait, across launches, until the host reads it.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <atomic>

#include "sp24_gemm.cuh"
#include "sp24_ptx.cuh"

namespace sp24 {
namespace {

// MMA kinds: 0 = f16 / bf16, 1 = int8, 2 = tf32, 3 = 8-bit floating point (e4m3 / e5m2)
__host__ __device__ constexpr bool one_byte_operands(int kind) { return kind == 1 || kind == 3; }

// Tall tiles (CTAS == 1, MBLK == kTallBlocks; sparse A, K-major B): up to 128 columns, two or three m-blocks (set
// per launch) that share each B box.  Their ring is finer: one slot per m-block and k-block (A and metadata) and
// a second ring for the B boxes, so that a slot is refilled as soon as its four MMAs are done.
constexpr int kTallBlocks = 3;
template <int CTAS, int MBLK>
constexpr bool is_tall = CTAS == 1 && MBLK == kTallBlocks;

// A cluster of CTAs may share the k-blocks of a tile (p.split_log): INT32 accumulators, which are the same in any order of the
// sums.  Kernels of their own (SPLIT): with it as a choice inside the others, short calls that do not split took up to 0.2 us
// (6 %) more.
template <int KIND, bool SPARSE, int CTAS, int MBLK, bool B_MN>
constexpr bool can_split = KIND == 1 && SPARSE && CTAS == 1 && MBLK == 1 && !B_MN;

template <int KIND, bool SPARSE, int BLOCK_N, int CTAS, int MBLK, bool B_MN>
struct Cfg {
  // 128-byte atoms per stage: sparse A is half as wide as B; the dense variant with two
  // m-blocks takes one atom per operand so that four stages still fit
  static constexpr int kBBoxes = SPARSE ? 2 : (MBLK == 2 ? 1 : 2);
  static constexpr int kABoxes = SPARSE ? 1 : kBBoxes;
  static constexpr int kABlockBytes = kABoxes * kBlockM * kAtomBytes;  // one m-block
  static_assert(MBLK == 1 || kABoxes == 1, "the m-blocks of a stage are one box of rows");
  static constexpr int kABytes = MBLK * kABlockBytes;
  static constexpr int kAtomElems = KIND == 0 ? 64 : (one_byte_operands(KIND) ? 128 : 32);  // elements per 128-byte row
  static constexpr int kKPerStage = kAtomElems * kBBoxes;  // logical K per stage
  // B with N contiguous (MN-major operand): 128-byte chunks along N, each kKPerStage k-rows of 128 bytes
  static constexpr int kBChunkElems = kAtomElems;
  static constexpr int kBChunkBytes = kKPerStage * kAtomBytes;
  static constexpr int kBKStepBytes = (SPARSE ? 2 : 1) * (kAtomElems / 4) * kAtomBytes;  // k-rows of one MMA
  // an MN-major tf32 operand exists only in the 128-byte swizzle with 32-byte units (groups of 4 k-rows)
  static constexpr uint32_t kBMnLayout = KIND == 2 ? ptx::kLayoutSw128Base32 : ptx::kLayoutSw128;
  static constexpr uint32_t kBMnSbo = KIND == 2 ? 512 : 1024;
  // A launch may use fewer columns than BLOCK_N (p.tile_n): rows of B (columns of D) a CTA loads per k-block, 128-byte
  // chunks of them (N contiguous), bytes
  __host__ __device__ static constexpr int b_rows(int tile_n) { return tile_n / CTAS; }
  __host__ __device__ static constexpr int b_chunks(int tile_n) { return (b_rows(tile_n) + kBChunkElems - 1) / kBChunkElems; }
  __host__ __device__ static constexpr int b_bytes(int tile_n) {
    return B_MN ? b_chunks(tile_n) * kBChunkBytes : kBBoxes * b_rows(tile_n) * kAtomBytes;
  }
  static constexpr int kEBlocks = SPARSE ? (one_byte_operands(KIND) ? 2 : 1) : 0;  // 2048-byte metadata blocks per m-block and stage
  static constexpr int kEBlockBytes = kEBlocks * 2048;
  static constexpr int kEBytes = MBLK * kEBlockBytes;
  static constexpr int kEAlloc = (kEBytes + 1023) / 1024 * 1024;
  __host__ __device__ static constexpr int stage_bytes(int tile_n) { return kABytes + b_bytes(tile_n) + kEAlloc; }
  // shared memory: [stage ring | epilogue staging | barriers]; 1 KB of slack for the 1024-byte alignment
  // The split between ring stages and epilogue staging is made per launch (the output type
  // decides how much staging is useful).
  static constexpr int kSmemLimit = 232448 - 1024 - 512;
  static constexpr int kMaxStages = 12;
  // stages of a ring of slots of `bytes`, the epilogue's staging beside them
  __host__ __device__ static constexpr int ring_stages(int bytes, int staging) {
    return (kSmemLimit - staging) / bytes > kMaxStages ? kMaxStages : (kSmemLimit - staging) / bytes;
  }
  // Epilogue form.  4-byte row-major outputs go through TMA boxes if every epilogue warp can have a
  // 4 KB box of its own without costing the ring of pairs a stage.  Everything else takes the warps' own loads and stores through a 2 KB transposing
  // buffer per warp (see epilogue_direct).
  __host__ __device__ static constexpr bool staged_epilogue(int cs, bool cols) {
    return CTAS == 2 && !cols && cs == 4 &&
           ring_stages(stage_bytes(BLOCK_N), kEpiWarps * 4096) == ring_stages(stage_bytes(BLOCK_N), kEpiWarps * 2048);
  }
  static constexpr int kAccStages = MBLK >= 2 ? 1 : ((2 * BLOCK_N + (SPARSE ? 32 : 0) <= (int)kTmemCols) ? 2 : 1);
  static constexpr int kECol = kAccStages * MBLK * BLOCK_N;        // first metadata column in tensor memory
  static constexpr int kMmasPerStage = SPARSE ? 4 : 4 * kBBoxes;   // per m-block and k-block
  // Stages of two k-blocks (p.kps; see the producer): A in whole 128-byte atoms, four k-blocks at least, and four such stages
  // in the ring (with three the ring is too coarse, us: bf16 64 x 6592 x 1408 7.0 -> 7.4, 2048 x 1024 x 2048 7.07 -> 7.22).
  // That is 16-bit and TF32 tiles of 32 columns, of 64 in a pair without a staged epilogue; 8-bit kinds, whose metadata is
  // twice as long, only in pairs of 32 columns.
  static constexpr bool kPairsOfKBlocks = SPARSE && !B_MN && MBLK == 1;
  static constexpr int k_blocks_of_a_stage(int tile_n, int staging, int64_t a_cols, bool conv) {
    return kPairsOfKBlocks && !conv && a_cols % kAtomElems == 0 && a_cols / kAtomElems >= 4 &&
                   ring_stages(2 * stage_bytes(tile_n), staging) >= 4 ? 2 : 1;
  }
  static constexpr int kSmemBytes = 232448;  // always the whole opt-in maximum
  static_assert(ring_stages(stage_bytes(BLOCK_N), kEpiWarps * 2048) >= 2, "need at least two stages");
  // the epilogue moves 32-column boxes; a last box of 16 columns (240-column tiles) is handled only by
  // epilogue_direct, which bounds every access by the tile's last column
  static_assert(BLOCK_N % 16 == 0, "tile width");
  static_assert(stage_bytes(32) % 1024 == 0 && stage_bytes(BLOCK_N) % 1024 == 0, "stages must keep the 1024-byte alignment of the atoms");
  static_assert(kECol + (SPARSE ? (is_tall<CTAS, MBLK> ? kMaxStages * 8 : 2 * MBLK * 8) : 0) <= (int)kTmemCols,
                "tensor memory overflow");
};

// Kernels with twelve epilogue warps beside the ones with eight (WARPS): int8 results of pairs, whose arithmetic is the longest,
// on a short K in several rounds of tiles, where it and not the main loop bounds a round.  Up to six k-blocks, us, device, eight
// warps and twelve: 3072 x 4096 x 256 10.3, 9.7; x 768 11.2, 10.6; x 1536 13.0, 12.4; 10944 x 5824 x 512 40.2, 37.1.  Not on a
// longer K (x 2048 14.3, 14.6) or in one round (288 x 4736 x 1344 5.4, 5.6); not for 16-bit results (4096 x 4096 x 768 12.5, 12.1
// but 9632 x 13344 x 416 70, 72, the stores bound it), other kinds (BERT FFN the same with twelve or sixteen) or wider tiles,
// whose ring would lose a stage.
template <int KIND, bool SPARSE, int BLOCK_N, int CTAS, int MBLK, bool B_MN>
constexpr bool twelve_warps = KIND == 1 && SPARSE && CTAS == 2 && MBLK == 1 && !B_MN && BLOCK_N == 224;

template <int KIND, bool SPARSE, int BLOCK_N, int CTAS, int MBLK, bool B_MN>
int epilogue_warps(const sp24_gemm_desc* d, int tile_n) {
  using C = Cfg<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN>;
  const int tile_m = kBlockM * CTAS * MBLK;
  return twelve_warps<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN> && elem_bytes(d->cd_type) == 1 && d->K <= 6 * C::kKPerStage &&
                 (d->M + tile_m - 1) / tile_m * ((d->N + tile_n - 1) / tile_n) > sm_count() / CTAS ? 12 : kEpiWarps;
}

struct Shared {
  uint64_t full[12], empty[12], tmem_full[2], tmem_empty[2];
  uint64_t split_full;             // the other CTAs' parts of the boxes that this one finishes are there
  uint64_t c_full[kEpiWarps][2];   // per epilogue warp and staging buffer: C box has landed
  uint32_t tmem_base;
  volatile uint32_t abort;
};
static_assert(sizeof(Shared) <= 512, "barrier block");

template <bool CLUSTER = false>  // (for what another CTA has written)
__device__ __forceinline__ bool bounded_wait(uint64_t* bar, uint32_t parity, Shared* sh, uint32_t* status,
                                             uint32_t code, long long limit) {
  auto try_wait = [&] { return CLUSTER ? ptx::mbar_try_wait_cluster(bar, parity) : ptx::mbar_try_wait(bar, parity); };
  // fast path: poll a while before any bookkeeping; try_wait itself suspends the thread briefly
#pragma unroll 1
  for (int i = 0; i < 64; ++i)
    if (try_wait()) return true;
  const long long t0 = clock64();
  uint32_t spins = 0;
  while (true) {
    if (try_wait()) return true;
    if ((++spins & 255u) == 0) {
      if (sh->abort) return false;
      if (clock64() - t0 > limit) {
        sh->abort = 1;
        atomicCAS(status, 0u, code);   // sticky: the first code stays until the host reads and clears it
        atomicAdd(status + 1, 1u);
        return false;
      }
    }
  }
}

// tile index -> (m_tile, n_tile): bands of `band_rows` m-tiles are swept n-tile by n-tile so that
// the tiles in flight at one time share a few A row-panels and B column-panels in the L2; every
// other band is swept from the last n-tile back, so that the first wave of a band uses the B
// columns the last wave of the band before has just read.
__device__ __forceinline__ void tile_coords(int t, const GemmParams& p, int& mt, int& nt) {
  const int band = p.by_band_tiles(t), in_band = t - band * (p.band * p.n_tiles);
  const int rows = min(p.band, p.m_tiles - band * p.band);
  nt = rows == p.band ? p.by_band(in_band) : p.by_last_band(in_band);
  mt = band * p.band + (in_band - nt * rows);
  if (band & 1) nt = p.n_tiles - 1 - nt;
}

template <int KIND>
__device__ __forceinline__ uint32_t make_idesc(bool sparse, bool b_mn_major, int a_fmt, int m, int n, bool acc_f16) {
  uint32_t d = 0;
  d |= (sparse ? 1u : 0u) << 2;
  d |= (KIND == 1 ? 2u : (acc_f16 ? 0u : 1u)) << 4;  // accumulator: int32 / fp32 / fp16
  // kind f16: f16 = 0, bf16 = 1; tf32: 2; int8: 1 = signed; 8-bit floats: e4m3 = 0, e5m2 = 1
  uint32_t fmt = (KIND == 0 || KIND == 3) ? (uint32_t)a_fmt : (KIND == 1 ? 1u : 2u);
  d |= fmt << 7;
  d |= fmt << 10;
  d |= (b_mn_major ? 1u : 0u) << 16;               // A is always K-major
  d |= (uint32_t)(n >> 3) << 17;
  d |= (uint32_t)(m >> 4) << 24;
  return d;                                        // no negate, no saturate
}

// Rows of A of a tile.  One m-block: rank 0 has the first 128 rows, rank 1 the next.  Two m-blocks: a CTA's
// blocks are neighbours (rank 0 rows 0-255 of the tile, rank 1 rows 256-511), so that one load brings
// both; in a last tile of at most 256 rows each CTA has one block instead of rank 0 having two.
template <int CTAS, int MBLK>
__device__ __forceinline__ int live_blocks(int mt, int M) {
  return MBLK != 2 ? 1 : (M - mt * (MBLK * CTAS * kBlockM) > CTAS * kBlockM ? 2 : 1);
}
template <int CTAS, int MBLK>
__device__ __forceinline__ int first_row(int mt, int cta_rank, int M) {
  static_assert(MBLK == 1 || (CTAS == 2 && MBLK == 2) || is_tall<CTAS, MBLK>, "tile shape");  // (tall: not used)
  return mt * (MBLK * CTAS * kBlockM) + cta_rank * kBlockM * live_blocks<CTAS, MBLK>(mt, M);
}

// ---- epilogue helpers ----------------------------------------------------------------------------
// Dequantising epilogue of the int8 path, all in fp32 and in exactly this order (the int8 output
// is compared bit for bit): t = float(acc) (round to nearest), y = fma(scale, t, bias), optional
// max(y, 0); int8 output: round-to-nearest-even of y * out_inv_scale, clamped to [-127, 127].
// (Two elements to an instruction where there is one.  The activation comes last: on the rounded code of an int8 output, on
// the packed values of a 16-bit one, which give what max before the rounding gives, NaN included.  Element by element, with
// both ends clamped and four bytes merged by logic, the epilogue was what int8 3072 x 4096 x 768 -> int8 waited for: us, device,
// 13.0 -> 11.5, in a loop of calls 12.75 -> 11.55; decoding 4096 x 32 x 4096 -> bf16 5.61 -> 5.53.)
__device__ __forceinline__ float2 dequant_pair(uint32_t acc0, uint32_t acc1, float scale, float bias) {
  return ptx::fma2(make_float2(__int2float_rn((int)acc0), __int2float_rn((int)acc1)), scale, make_float2(bias, bias));
}
// Four int8 codes of a word, at least `low`: -127, or 0 after the activation.
__device__ __forceinline__ uint32_t requant_word(float2 y01, float2 y23, float inv, int low) {
  const float2 v01 = ptx::mul2(y01, inv), v23 = ptx::mul2(y23, inv);
  const int q0 = max(__float2int_rn(v01.x), low), q1 = max(__float2int_rn(v01.y), low);
  const int q2 = max(__float2int_rn(v23.x), low), q3 = max(__float2int_rn(v23.y), low);
  return ptx::pack_sat_s8(q1, q0, ptx::pack_sat_s8(q3, q2, 0));
}

__device__ __forceinline__ uint32_t pack_16bit(float lo, float hi, bool bf) {
  if (bf) {
    __nv_bfloat162 o = __float22bfloat162_rn(make_float2(lo, hi));
    return *reinterpret_cast<uint32_t*>(&o);
  }
  __half2 o = __float22half2_rn(make_float2(lo, hi));
  return *reinterpret_cast<uint32_t*>(&o);
}
__device__ __forceinline__ uint32_t relu_16bit(uint32_t w, bool bf) {
  if (bf) {
    const __nv_bfloat162 o = __hmax2(*reinterpret_cast<const __nv_bfloat162*>(&w), __nv_bfloat162(__ushort_as_bfloat16(0), __ushort_as_bfloat16(0)));
    return *reinterpret_cast<const uint32_t*>(&o);
  }
  const __half2 o = __hmax2(*reinterpret_cast<const __half2*>(&w), __half2(__ushort_as_half(0), __ushort_as_half(0)));
  return *reinterpret_cast<const uint32_t*>(&o);
}
__device__ __forceinline__ float2 unpack_16bit(uint32_t w, bool bf) {
  return bf ? __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162*>(&w))
            : __half22float2(*reinterpret_cast<const __half2*>(&w));
}

// One thread's row of a box of `cols` columns: out = alpha * acc + beta * c (or the dequantising form) as
// the packed words of the output row (CS bytes an element; CS = 1 is always the dequantising form).
// `c` holds the row's C values in the same packing and is read only if has_c.  One multiply and
// one fused multiply-add per element, whichever path stores the row.
template <int KIND, int CS, int COLUMNS>
__device__ __forceinline__ void compute_row(const uint32_t (&r)[COLUMNS], const uint32_t (&c)[COLUMNS * CS / 4], bool has_c,
                                            const GemmParams& p, float scale, float bias, uint32_t (&o)[COLUMNS * CS / 4]) {
  if constexpr (CS == 1) {
    const int low = p.relu ? 0 : -127;
#pragma unroll
    for (int e = 0; e < COLUMNS / 4; ++e)
      o[e] = requant_word(dequant_pair(r[4 * e], r[4 * e + 1], scale, bias), dequant_pair(r[4 * e + 2], r[4 * e + 3], scale, bias),
                          p.out_inv_scale, low);
  } else if constexpr (CS == 4) {
    if (KIND == 1 && p.dequant) {
#pragma unroll
      for (int e = 0; e < COLUMNS; e += 2) {
        const float2 y = dequant_pair(r[e], r[e + 1], scale, bias);
        o[e] = __float_as_uint(y.x);
        o[e + 1] = __float_as_uint(y.y);
      }
      if (p.relu) {
#pragma unroll
        for (int e = 0; e < COLUMNS; ++e) o[e] = __float_as_uint(fmaxf(__uint_as_float(o[e]), 0.f));
      }
    } else if (KIND == 1) {
#pragma unroll
      for (int e = 0; e < COLUMNS; ++e) o[e] = r[e] + (has_c ? c[e] : 0u);
    } else {
#pragma unroll
      for (int e = 0; e < COLUMNS; e += 2) {
        float2 f = ptx::mul2(make_float2(__uint_as_float(r[e]), __uint_as_float(r[e + 1])), p.alpha);
        if (has_c) f = ptx::fma2(make_float2(__uint_as_float(c[e]), __uint_as_float(c[e + 1])), p.beta, f);
        o[e] = __float_as_uint(f.x);
        o[e + 1] = __float_as_uint(f.y);
      }
    }
  } else {
    auto pack = [&](bool bf) {
#pragma unroll
      for (int e = 0; e < COLUMNS / 2; ++e) {
        float2 f;
        if (KIND == 1) {  // dequantised to a 16-bit type (the plain int8 GEMM writes 4-byte results)
          f = dequant_pair(r[2 * e], r[2 * e + 1], scale, bias);
        } else {
          f = ptx::mul2(make_float2(__uint_as_float(r[2 * e]), __uint_as_float(r[2 * e + 1])), p.alpha);
          if (has_c) f = ptx::fma2(unpack_16bit(c[e], bf), p.beta, f);
        }
        o[e] = pack_16bit(f.x, f.y, bf);
      }
      if (KIND == 1 && p.relu) {
#pragma unroll
        for (int e = 0; e < COLUMNS / 2; ++e) o[e] = relu_16bit(o[e], bf);
      }
    };
    if (p.cd_type == SP24_BF16) pack(true);
    else pack(false);
  }
}

// FP16 accumulation: every accumulator cell of tensor memory holds a binary16 value in its low half
template <int COLUMNS>
__device__ __forceinline__ void widen_f16_accumulators(uint32_t (&r)[COLUMNS]) {
#pragma unroll
  for (int e = 0; e < COLUMNS; ++e) r[e] = __float_as_uint(__half2float(__ushort_as_half((unsigned short)(r[e] & 0xFFFFu))));
}

// TMA-staged form of a 4-byte row-major box (rows of 128 bytes in the TMA's 128-byte swizzle: 16-byte
// unit v of row r sits at unit v ^ (r & 7), which also keeps the row-per-thread accesses free of bank
// conflicts): C, if any, is in the staging buffer; the result replaces it there.
template <int KIND, bool HAS_C>
__device__ __forceinline__ void convert_row_staged(const uint32_t (&r)[32], uint8_t* buf, int lane, const GemmParams& p,
                                                   float scale, float bias) {
  uint32_t c[32], o[32];
  uint8_t* row = buf + lane * 128;
  if (HAS_C) {
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint4 x = *reinterpret_cast<const uint4*>(row + ((v ^ (lane & 7)) << 4));
      c[4 * v] = x.x; c[4 * v + 1] = x.y; c[4 * v + 2] = x.z; c[4 * v + 3] = x.w;
    }
  }
  compute_row<KIND, 4, 32>(r, c, HAS_C, p, scale, bias, o);
#pragma unroll
  for (int v = 0; v < 8; ++v)
    *reinterpret_cast<uint4*>(row + ((v ^ (lane & 7)) << 4)) = make_uint4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
}

// ---- epilogue in which the warps move C and D themselves -----------------------------------------
// What bounds it is how fast eight warps get through their instructions, not the stores: with the boxes of a tile
// unrolled into straight code a box took a warp 1700 cycles (one pair of CTAs alone on the chip or all of them, the
// same), a third of them waiting for instructions that were fetched for this one box, and two warps on a scheduler
// cannot hide that.  So: one short loop over the boxes that exist, with C a loop of four, shared-memory accesses in
// groups so that they overlap, packed FP32 arithmetic.  Cycles from the accumulators of a 512 x 224 tile being complete
// to their hand-back, unrolled and now (timestamps included): 16-bit results 12,700 and 5,800, with C 18,400 and 9,600,
// column-major 14,800 and 6,300, with C 20,800 and 9,500.  (Where more than eight warps pay: twelve_warps.)
// A box is 32 rows x 64 bytes of output (32 columns, 16 of a 4-byte type; 32 bytes of a 1-byte type).  Per box: the
// accumulators of this thread's row come out of tensor memory (loaded while the box before is stored), are converted
// in registers and stored by way of a 2 KB buffer of the warp.
// Row-major outputs: the rows are written to the buffer and read back transposed, so that the global stores of a warp
// cover whole 64-byte row segments.
// Column-major outputs (D stored [N][M], M contiguous): the lanes of a warp hold 32 consecutive m of
// each column, so a 4-byte box is stored straight from registers, one 128-byte line per column; the
// 1- and 2-byte boxes are transposed on the way out of the same per-warp buffer by ldmatrix.trans.
// The eight rows of ldmatrix matrix i are m = 8 j + 2 i + b (j = 0..3, b = 0, 1), which leaves each
// thread with eight consecutive m of one column (2-byte) or of two columns (1-byte): 16- and 8-byte
// stores.  16-byte unit u of buffer row m sits at u ^ (((m >> 1) ^ (m >> 3)) & 3): no bank conflicts
// in the row-wise writes, the ldmatrix reads and the row-wise reads of 64-byte rows (those of 1-byte boxes,
// half as wide, meet in pairs).
// C is loaded in the order of the stores (whole 64-byte row segments as well) into registers, four boxes ahead, the
// first four of a tile before its accumulators are complete, and goes to the rows' owners through the buffer.
template <int KIND, int CS, bool COLS, bool HAS_C, int BLOCK_N, int CTAS, int MBLK, int ACC_STAGES, int WARPS, bool SPLIT>
__device__ __forceinline__ void epilogue_direct(const GemmParams& p, Shared* sh, uint8_t* epi, uint32_t tmem_base,
                                              int cta_rank, int cluster_id, int num_clusters, int num_tiles, int warp,
                                              int lane, uint32_t parts, int split_rank) {
  constexpr int kCols = CS == 4 ? 16 : 32;  // columns of a box
  constexpr int W = kCols * CS / 4;         // 32-bit words of one box row
  constexpr int P = 4;                      // boxes whose C values are held in registers
  constexpr int kUnits = W / 4;             // 16-byte units of a buffer row that hold data
  constexpr int kUnitElems = 16 / CS;       // elements per 16-byte unit
  constexpr int kRowsPerStore = 32 / kUnits;
  const int q = warp & 3, turn = (warp - kFirstEpiWarp) >> 2;  // lane quarter, and first box of this warp there
  uint8_t* stage = epi + (warp - kFirstEpiWarp) * 2048;
  const uint8_t* Cb = static_cast<const uint8_t*>(p.C);
  uint8_t* Db = static_cast<uint8_t*>(p.D);
  const size_t ldc_b = (size_t)p.ldc * CS, ldd_b = (size_t)p.ldd * CS;
  const int M = (int)p.M, N = (int)p.N;
  constexpr bool has_c = HAS_C;
  // this lane's row of the buffer, its unit 0 under the swizzle (xor the unit into bits 4..5) ...
  const uint32_t own_row = ptx::smem_u32(stage) + (uint32_t)(lane * 64 + ((((lane >> 1) ^ (lane >> 3)) & 3) << 4));
  // ... for ldmatrix / stmatrix ...
  const int tm_i = lane >> 3, tm_j = (lane & 7) >> 1;
  const uint32_t tm_row = ptx::smem_u32(stage) + (uint32_t)((8 * tm_j + 2 * tm_i + (lane & 1)) * 64 + ((tm_i ^ tm_j) << 4));
  // ... and in the order of row-major stores: this lane's row and unit of the first store (of the next ones: kRowsPerStore
  // rows on)
  const int st_r = lane / kUnits, st_u = lane % kUnits;
  const uint32_t st_row = ptx::smem_u32(stage) + (uint32_t)(st_r * 64 + ((st_u ^ (((st_r >> 1) ^ (st_r >> 3)) & 3)) << 4));
  // K-blocks shared by a cluster of CTAs: the boxes of warp w are finished by CTA w mod the cluster's size.  The other CTAs'
  // warps w send it their accumulators of these boxes (16-byte units of 32 lanes) into shared memory kept for them; it adds
  // them up as it takes a box from its own tensor memory.
  const int split_log = SPLIT ? p.split_log : 0, split = 1 << split_log;
  const int owner = (warp - kFirstEpiWarp) & (split - 1);
  const bool mine = owner == split_rank;
  const int warp_boxes = (p.tile_n / kCols + 1) / 2, owner_boxes = (kEpiWarps >> split_log) * warp_boxes;  // (room for)
  auto part_of = [&](int from_rank, int sc) {
    const int i = ((from_rank - owner - 1) & (split - 1)) * owner_boxes + ((warp - kFirstEpiWarp) >> split_log) * warp_boxes + (sc >> 1);
    return parts + (uint32_t)(i * (kCols * 128) + lane * 16);
  };
  auto st_addr = [&](int k) { return (st_row ^ (uint32_t)(((k * kRowsPerStore) >> 3) << 4)) + k * kRowsPerStore * 64; };
  int acc = 0;
  uint32_t acc_phase = 0;
  for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
    int mt, nt;
    tile_coords(t, p, mt, nt);
    const int tile_col = nt * p.tile_n, col_end = min(N, tile_col + p.tile_n);  // columns of this tile stop here
    // the boxes of this lane quarter: `nsub` in a row, `blocks` rows of them (m-blocks); the warps take them in turn
    const int row_q = (is_tall<CTAS, MBLK> ? mt * p.mblk * kBlockM : first_row<CTAS, MBLK>(mt, cta_rank, M)) + q * 32;
    const int nsub = (col_end - tile_col + kCols - 1) / kCols;
    const int blocks = min(is_tall<CTAS, MBLK> ? p.mblk : live_blocks<CTAS, MBLK>(mt, M), (M - row_q + kBlockM - 1) / kBlockM);
    auto step = [&](int& j, int& sc, int by) {
      sc += by;
      while (sc >= nsub) { sc -= nsub; ++j; }
    };
    int j = 0, sc = 0;  // the box at hand
    step(j, sc, turn);
    // C values of a box, in the order of the stores
    auto load_c = [&](int row0, int col0, uint32_t (&c)[W]) {
      if constexpr (CS == 1) {
      } else if constexpr (!COLS) {
        const int col = col0 + st_u * kUnitElems;
        const uint8_t* src = Cb + (size_t)(row0 + st_r) * ldc_b + (size_t)col * CS;
#pragma unroll
        for (int k = 0; k < kUnits; ++k) {
          if (col < col_end && row0 + st_r + k * kRowsPerStore < M) {
            const uint4 x = *reinterpret_cast<const uint4*>(src + k * kRowsPerStore * ldc_b);
            c[4 * k] = x.x; c[4 * k + 1] = x.y; c[4 * k + 2] = x.z; c[4 * k + 3] = x.w;
          }
        }
      } else if constexpr (CS == 2) {
        const int m = row0 + 8 * (lane & 3);
        const uint8_t* src = Cb + (size_t)(col0 + (lane >> 2)) * ldc_b + (size_t)m * CS;
#pragma unroll
        for (int nb = 0; nb < 4; ++nb) {
          if (m < M && col0 + 8 * nb + (lane >> 2) < col_end) {
            const uint4 x = *reinterpret_cast<const uint4*>(src + 8 * nb * ldc_b);
            c[4 * nb] = x.x; c[4 * nb + 1] = x.y; c[4 * nb + 2] = x.z; c[4 * nb + 3] = x.w;
          }
        }
      } else if (row0 + lane < M) {
        const uint8_t* src = Cb + (size_t)col0 * ldc_b + (size_t)(row0 + lane) * CS;
#pragma unroll
        for (int e = 0; e < kCols; ++e)
          if (col0 + e < col_end) c[e] = *reinterpret_cast<const uint32_t*>(src + e * ldc_b);
      }
    };
    // C from the order of the stores to the rows' owners (4-byte column-major boxes are with them already)
    auto share_c = [&](uint32_t (&c)[W]) {
      if constexpr (CS == 1 || (CS == 4 && COLS)) return;
      __syncwarp();  // the reads of the box before are done
#pragma unroll
      for (int k = 0; k < kUnits; ++k) {
        if constexpr (COLS) ptx::stmatrix_x4_trans(tm_row ^ (uint32_t)(k << 4), c[4 * k], c[4 * k + 1], c[4 * k + 2], c[4 * k + 3]);
        else ptx::st_shared_v4(st_addr(k), c[4 * k], c[4 * k + 1], c[4 * k + 2], c[4 * k + 3]);
      }
      __syncwarp();
#pragma unroll
      for (int u = 0; u < kUnits; ++u)
        ptx::ld_shared_v4(own_row ^ (uint32_t)(u << 4), c[4 * u], c[4 * u + 1], c[4 * u + 2], c[4 * u + 3]);
    };
    // packed output rows -> D
    auto store = [&](const uint32_t (&o)[W], int row0, int col0) {
      if constexpr (CS == 4 && COLS) {
        if (row0 + lane < M) {
          uint8_t* dst = Db + (size_t)col0 * ldd_b + (size_t)(row0 + lane) * CS;
#pragma unroll
          for (int e = 0; e < kCols; ++e)
            if (col0 + e < col_end) *reinterpret_cast<uint32_t*>(dst + e * ldd_b) = o[e];
        }
      } else {
        if (!has_c) __syncwarp();  // the reads of the box before are done (with C each lane writes what it alone has read)
#pragma unroll
        for (int u = 0; u < kUnits; ++u)
          ptx::st_shared_v4(own_row ^ (uint32_t)(u << 4), o[4 * u], o[4 * u + 1], o[4 * u + 2], o[4 * u + 3]);
        __syncwarp();
        if constexpr (COLS) {
          const int m = row0 + 8 * (lane & 3);
          const int n1 = col0 + (CS == 2 ? 1 : 2) * (lane >> 2);
          uint8_t* dst = Db + (size_t)n1 * ldd_b + (size_t)m * CS;
          uint32_t x[kUnits][4];
#pragma unroll
          for (int nb = 0; nb < kUnits; ++nb) ptx::ldmatrix_x4_trans(tm_row ^ (uint32_t)(nb << 4), x[nb][0], x[nb][1], x[nb][2], x[nb][3]);
#pragma unroll
          for (int nb = 0; nb < kUnits; ++nb) {
            const uint32_t(&w)[4] = x[nb];
            if (m < M && n1 + nb * (16 / CS) < col_end) {
              uint8_t* at = dst + nb * (16 / CS) * ldd_b;
              if constexpr (CS == 2) {
                *reinterpret_cast<uint4*>(at) = make_uint4(w[0], w[1], w[2], w[3]);
              } else {
                // 16-bit units hold two neighbouring columns: split them
                *reinterpret_cast<uint2*>(at) = make_uint2(__byte_perm(w[0], w[1], 0x6420), __byte_perm(w[2], w[3], 0x6420));
                *reinterpret_cast<uint2*>(at + ldd_b) =
                    make_uint2(__byte_perm(w[0], w[1], 0x7531), __byte_perm(w[2], w[3], 0x7531));
              }
            }
          }
        } else {
          const int col = col0 + st_u * kUnitElems;
          uint8_t* dst = Db + (size_t)(row0 + st_r) * ldd_b + (size_t)col * CS;
          uint4 x[kUnits];
#pragma unroll
          for (int k = 0; k < kUnits; ++k) ptx::ld_shared_v4(st_addr(k), x[k].x, x[k].y, x[k].z, x[k].w);
#pragma unroll
          for (int k = 0; k < kUnits; ++k)
            if (col < col_end && row0 + st_r + k * kRowsPerStore < M)
              *reinterpret_cast<uint4*>(dst + k * kRowsPerStore * ldd_b) = x[k];
        }
      }
    };
    auto hand_back = [&] {  // this warp's part of the accumulators is in registers: the MMA issuer (CTA 0 of the pair) may go on
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CTAS == 1) ptx::mbar_arrive(&sh->tmem_empty[acc]);
        else ptx::mbar_arrive_cluster(&sh->tmem_empty[acc], 0);
      }
    };
    const uint32_t t_acc = tmem_base + (acc * MBLK) * BLOCK_N + ((uint32_t)(q * 32) << 16);
    uint32_t r[kCols], creg[P][W];
    float scale = 1.f, bias = 0.f;
    auto load_scale = [&](int row0) {
      if (KIND == 1 && p.dequant) {
        const int row = min(row0 + lane, M - 1);
        scale = p.row_scale[row];
        bias = p.bias ? p.bias[row] : 0.f;
      }
    };
    // One box, with the C values in c; true if there is another one.
    int cj = j, csc = sc;  // has_c: the next box whose C values are fetched
    auto fetch_c = [&](uint32_t (&c)[W]) {
      if (cj < blocks) load_c(row_q + cj * kBlockM, tile_col + csc * kCols, c);
      step(cj, csc, WARPS / 4);
    };
    auto box = [&](uint32_t (&c)[W]) -> bool {
      const int row0 = row_q + j * kBlockM, col0 = tile_col + sc * kCols, j0 = j, sc0 = sc;
      step(j, sc, WARPS / 4);
      const bool more = j < blocks;
      uint32_t o[W];
      if (has_c) share_c(c);
      ptx::tmem_ld_wait(r);
      if (!more) hand_back();
      if constexpr (SPLIT) {
#pragma unroll 1
        for (int i = 1; i < split; ++i) {
          const uint32_t from = part_of(split_rank + i, sc0);
#pragma unroll
          for (int u = 0; u < kCols / 4; ++u) {
            uint32_t x[4];
            ptx::ld_shared_v4(from + u * 512, x[0], x[1], x[2], x[3]);
            r[4 * u] += x[0]; r[4 * u + 1] += x[1]; r[4 * u + 2] += x[2]; r[4 * u + 3] += x[3];
          }
        }
      }
      if (KIND == 0 && p.acc_f16) widen_f16_accumulators(r);
      compute_row<KIND, CS, kCols>(r, c, has_c, p, scale, bias, o);
      if (more) {
        ptx::tmem_ld_32x32b(t_acc + j * BLOCK_N + sc * kCols, r);
        if (j != j0) load_scale(row_q + j * kBlockM);
      }
      if (has_c) fetch_c(c);
      store(o, row0, col0);
      return more;
    };
    const bool any = mine && j < blocks;
    if (any) load_scale(row_q + j * kBlockM);
    if (has_c && mine) {
#pragma unroll
      for (int n = 0; n < P; ++n) fetch_c(creg[n]);
    }
    const long long limit = SPLIT && p.test_skip_stage == 2 + split_rank ? 4 * p.wait_limit : p.wait_limit;  // (as in gemm_kernel)
    if (!bounded_wait(&sh->tmem_full[acc], acc_phase, sh, p.status, 4u, limit)) break;
    ptx::tc_fence_after();
    if constexpr (SPLIT) {
      if (!mine) {
        const uint32_t bar = ptx::map_to_cta(ptx::smem_u32(&sh->split_full), (uint32_t)owner);
#pragma unroll 1
        for (; j < blocks; step(j, sc, WARPS / 4)) {
          const uint32_t to = ptx::map_to_cta(part_of(split_rank, sc), (uint32_t)owner);
          ptx::tmem_ld_32x32b(t_acc + sc * kCols, r);
          ptx::tmem_ld_wait(r);
#pragma unroll
          for (int u = 0; u < kCols / 4; ++u) ptx::st_async_v4(to + u * 512, r[4 * u], r[4 * u + 1], r[4 * u + 2], r[4 * u + 3], bar);
        }
      } else {
        if (lane == 0) {
          const int boxes = blocks > 0 && nsub > turn ? (nsub - turn + 1) / 2 : 0;
          ptx::mbar_expect_tx(&sh->split_full, (uint32_t)(boxes * (split - 1) * kCols * 128));
        }
        if (!bounded_wait<true>(&sh->split_full, 0, sh, p.status, 6u, p.wait_limit)) break;
      }
    }
    if (!any) {
      hand_back();
    } else {
      ptx::tmem_ld_32x32b(t_acc + j * BLOCK_N + sc * kCols, r);
      if (!has_c) {
#pragma unroll 1
        while (box(creg[0])) {
        }
      } else {
        bool more = true;
#pragma unroll 1
        while (more) {
#pragma unroll
          for (int n = 0; n < P; ++n)
            if (more) more = box(creg[n]);
        }
      }
    }
    if (++acc == ACC_STAGES) { acc = 0; acc_phase ^= 1u; }
  }
}

// CS, COLS, HAS_C: bytes of an output element, column-major output, C is added.  A kernel for each form of the output, so that
// it holds one epilogue: with all of them behind branches of one kernel, a tile's epilogue took up to twice as long whatever
// the form (us, branches -> own kernels: bf16 24576 x 224 x 4096 with 512 x 224 tiles 39.8 -> 34.3, with C 43.6 -> 37.8).  With
// and without C apart (the registers of four boxes of it): f16 256 x 256 x 512 3.29 -> 3.19, BERT FFN 12.48 -> 12.26, bf16
// 8480 x 896 x 384 7.83 -> 7.46, with C 9920 x 544 x 1216 16.1 -> 15.6, f16 1184 x 736 x 1008 5.92 -> 5.82; none slower.
template <int KIND, bool SPARSE, int BLOCK_N, int CTAS, int MBLK, bool B_MN, int CS, bool COLS, bool HAS_C, bool SPLIT = false, int WARPS = kEpiWarps>
__global__ void __launch_bounds__(32 * (kFirstEpiWarp + WARPS), 1)
gemm_kernel(const __grid_constant__ CUtensorMap map_a, const __grid_constant__ CUtensorMap map_b,
            const __grid_constant__ CUtensorMap map_e, const __grid_constant__ CUtensorMap map_c,
            const __grid_constant__ CUtensorMap map_d, const GemmParams p) {
  using C = Cfg<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN>;
  extern __shared__ uint8_t smem_raw[];
  // Operand atoms need 1024-byte alignment for the 128-byte swizzle.
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  constexpr bool kTall = is_tall<CTAS, MBLK>;
  static_assert(!kTall || (SPARSE && !B_MN && C::kABoxes == 1 && C::kBBoxes == 2), "tall tiles: sparse A, K-major B");
  // tall tiles: [slots of A and metadata | slots of B | epilogue staging]
  const int tile_n = p.tile_n, b_bytes = C::b_bytes(tile_n), b_slot_bytes = kTall ? b_bytes : 0;
  const int kps = C::kPairsOfKBlocks ? p.kps : 1;  // k-blocks of a stage
  const int slot_bytes = kTall ? C::kABlockBytes + C::kEBlockBytes : kps * (C::kABytes + b_bytes + C::kEAlloc);
  uint8_t* b_ring = smem + p.stages * slot_bytes;
  uint8_t* epi = b_ring + (kTall ? p.b_stages * b_slot_bytes : SPLIT ? p.part_bytes : 0);
  Shared* sh = reinterpret_cast<Shared*>(epi + p.epi_bytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t cta_rank = CTAS == 2 ? ptx::cluster_ctarank() : 0;
  static_assert(WARPS == kEpiWarps || !(SPLIT || C::staged_epilogue(CS, COLS)), "these count on eight epilogue warps");
  static_assert(!SPLIT || can_split<KIND, SPARSE, CTAS, MBLK, B_MN>, "only INT32 sums may be split");
  const int split_log = SPLIT ? p.split_log : 0, split_rank = SPLIT ? (int)ptx::cluster_ctarank() : 0;
  const int cluster_id = SPLIT ? blockIdx.x >> split_log : blockIdx.x / CTAS;
  const int num_clusters = SPLIT ? gridDim.x >> split_log : gridDim.x / CTAS;
  // this CTA's k-blocks
  const int kb_begin = SPLIT ? (p.k_blocks * split_rank) >> split_log : 0;
  const int kb_end = SPLIT ? (p.k_blocks * (split_rank + 1)) >> split_log : p.k_blocks;
  const int num_tiles = p.m_tiles * p.n_tiles;
  // (test hook: the CTA whose k-block is left out waits longer, so that the others' waits for its sums are the first to expire)
  auto wait_limit = [&] { return SPLIT && p.test_skip_stage == 2 + split_rank ? 4 * p.wait_limit : p.wait_limit; };

  // Set-up: lanes of a warp initialise the barriers, and the pair meets without a release.  All that a CTA of a pair has
  // to know before it goes on is that the peer's barriers are there, and fence.mbarrier_init publishes those; that the
  // peer has its tensor memory follows from its loads, which it issues after that.  With one thread for all barriers and
  // a releasing cluster barrier (1040 cycles) the pair was ready 1990 cycles after its start, now 1240 (BERT FFN, device,
  // with the tile coordinates by multiplication: 12.8 -> 11.9 us).
  if (warp == 0) {
    if (lane < p.stages) {
      ptx::mbar_init(&sh->full[lane], 1);
      ptx::mbar_init(&sh->empty[lane], 1);
    }
    if (lane < 2) {
      ptx::mbar_init(&sh->tmem_full[lane], 1);
      ptx::mbar_init(&sh->tmem_empty[lane], WARPS * CTAS);  // one arrival per epilogue warp of the pair
    }
    if (C::staged_epilogue(CS, COLS) && lane < 2 * kEpiWarps) ptx::mbar_init(&sh->c_full[lane >> 1][lane & 1], 1);
    if (SPLIT && lane == 0) ptx::mbar_init(&sh->split_full, kEpiWarps >> split_log);
    if (lane == 0) sh->abort = 0;
    ptx::fence_barrier_init();
    __syncwarp();
  }
  if (CTAS == 2 || SPLIT) ptx::cluster_arrive_relaxed();
  if (warp == 1) {
    ptx::tmem_alloc<CTAS>(&sh->tmem_base, kTmemCols);
    ptx::tmem_relinquish<CTAS>();
  } else if (threadIdx.x == 0) {
    ptx::prefetch_tensormap(&map_a);
    ptx::prefetch_tensormap(&map_b);
    if (SPARSE) ptx::prefetch_tensormap(&map_e);
    if (C::staged_epilogue(CS, COLS)) {
      if (HAS_C) ptx::prefetch_tensormap(&map_c);
      ptx::prefetch_tensormap(&map_d);
    }
  }
  ptx::tc_fence_before();
  __syncthreads();
  if (CTAS == 2) ptx::cluster_wait();
  ptx::tc_fence_after();
  const uint32_t tmem_base = sh->tmem_base;
  let_next_start();
  wait_for_stream();

  // tall tiles: m-blocks of tile row mt that have rows (the rest are neither loaded nor multiplied) ...
  auto tall_live = [&](int mt) -> int { return min(p.mblk, ((int)p.M - mt * p.mblk * kBlockM + kBlockM - 1) / kBlockM); };
  // ... and the slots of a CTA's ring.  B's slots have no barriers of their own: the box of k-block kb lands with
  // the k-block's first m-block, and with at most (b_stages - 1) * (m-blocks of a tile) + 1 slots that m-block's
  // slot is free only when all of k-block kb - b_stages has been multiplied.
  auto tall_slots = [&]() -> int {
    const bool has_last = cluster_id == (p.m_tiles - 1) % num_clusters || p.n_tiles > 1;  // the last tile row may have fewer
    return min(p.stages, (p.b_stages - 1) * (has_last ? tall_live(p.m_tiles - 1) : p.mblk) + 1);
  };

  if (kTall && warp == 0) {
    // ------------------------------ TMA producer, tall tiles ------------------------------
    if (ptx::elect_one()) {
      int slot = 0, b_slot = 0;
      uint32_t phase = 0;
      const int slots = tall_slots();
      const uint32_t ring = ptx::smem_u32(smem), b_ring_addr = ptx::smem_u32(b_ring), full0 = ptx::smem_u32(&sh->full[0]);
      for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
        int mt, nt;
        tile_coords(t, p, mt, nt);
        const int live = tall_live(mt), blk0 = mt * p.mblk;
        bool ok = true;
        for (int kb = 0; kb < p.k_blocks && ok; ++kb) {
#pragma unroll
          for (int j = 0; j < MBLK; ++j) {
            if (j >= live) break;
            if (!(ok = bounded_wait(&sh->empty[slot], phase ^ 1u, sh, p.status, 1u, p.wait_limit))) break;
            const uint32_t full = full0 + 8 * slot, sa = ring + slot * slot_bytes;
            // (test hook: the slot is neither armed nor loaded, so that the issuer's wait for it expires)
            if (!(j == 0 && p.test_skip_stage && t == cluster_id && kb == 1)) {
              ptx::mbar_expect_tx(&sh->full[slot], (uint32_t)(slot_bytes + (j == 0 ? b_slot_bytes : 0)));
              if (j == 0) {
                const uint32_t sb = b_ring_addr + b_slot * b_slot_bytes;
                if (p.b_3d) {
                  ptx::tma_load_3d<1>(sb, &map_b, full, 0, nt * tile_n, kb * C::kBBoxes);
                } else {
#pragma unroll
                  for (int i = 0; i < C::kBBoxes; ++i)
                    ptx::tma_load_2d<1>(sb + i * tile_n * kAtomBytes, &map_b, full, (kb * C::kBBoxes + i) * C::kAtomElems,
                                        nt * tile_n);
                }
              }
              ptx::tma_load_2d<1>(sa, &map_a, full, kb * C::kAtomElems, (blk0 + j) * kBlockM);
              ptx::tma_load_3d<1>(sa + C::kABlockBytes, &map_e, full, 0, 16 * kb * C::kEBlocks, blk0 + j);
            }
            if (++slot == slots) { slot = 0; phase ^= 1u; }
          }
          if (++b_slot == p.b_stages) b_slot = 0;
        }
      }
    }
  } else if (kTall && warp == 1) {
    // ------------------------------ MMA issuer, tall tiles ------------------------------
    if (ptx::elect_one()) {
      int slot = 0, b_slot = 0;
      uint32_t phase = 0, acc_phase = 0;
      const int slots = tall_slots();
      const uint32_t ring = ptx::smem_u32(smem), b_ring_addr = ptx::smem_u32(b_ring), b_atom = tile_n * kAtomBytes;
      for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
        int mt, nt;
        tile_coords(t, p, mt, nt);
        const int live = tall_live(mt);
        const uint32_t idesc = make_idesc<KIND>(SPARSE, false, p.a_fmt, kBlockM, min(tile_n, (int)p.N - nt * tile_n),
                                                KIND == 0 && p.acc_f16);
        if (!bounded_wait(&sh->tmem_empty[0], acc_phase ^ 1u, sh, p.status, 2u, p.wait_limit)) break;
        ptx::tc_fence_after();
        bool ok = true;
        for (int kb = 0; kb < p.k_blocks && ok; ++kb) {
          const uint64_t db0 = ptx::smem_desc(b_ring_addr + b_slot * b_slot_bytes, ptx::kLayoutSw128, 1024);
#pragma unroll
          for (int j = 0; j < MBLK; ++j) {
            if (j >= live) break;
            if (!(ok = bounded_wait(&sh->full[slot], phase, sh, p.status, 3u, p.wait_limit))) break;
            ptx::tc_fence_after();
            // (metadata columns per slot: a full slot also says that nothing reads its columns any more)
            const uint32_t sa = ring + slot * slot_bytes, e_tmem = tmem_base + C::kECol + slot * 8, d_tmem = tmem_base + j * BLOCK_N;
#pragma unroll
            for (int i = 0; i < C::kEBlocks; ++i)
              ptx::tmem_cp_128x128b<CTAS>(e_tmem + 4 * i, ptx::smem_desc(sa + C::kABlockBytes + i * 2048, ptx::kLayoutNone, 128));
            const uint64_t da0 = ptx::smem_desc(sa, ptx::kLayoutSw128, 1024);
#pragma unroll
            for (int k = 0; k < C::kMmasPerStage; ++k) {
              // the address fields of the descriptors count 16-byte units
              const uint64_t da = da0 + (k * 32 >> 4), db = db0 + (((k >> 1) * b_atom + (k & 1) * 64) >> 4);
              const uint32_t accumulate = (kb > 0 || k > 0) ? 1u : 0u;
              if (!one_byte_operands(KIND))
                ptx::mma_sparse<KIND, CTAS>(d_tmem, da, db, e_tmem + (k & ~1), idesc | (uint32_t)(k & 1), accumulate);
              else
                ptx::mma_sparse<KIND, CTAS>(d_tmem, da, db, e_tmem + 2 * k, idesc, accumulate);
            }
            ptx::tc_commit(&sh->empty[slot]);
            if (++slot == slots) { slot = 0; phase ^= 1u; }
          }
          if (++b_slot == p.b_stages) b_slot = 0;
        }
        if (!ok) break;
        ptx::tc_commit(&sh->tmem_full[0]);
        acc_phase ^= 1u;
      }
    }
  } else if (warp == 0) {
    // ------------------------------ TMA producer ------------------------------
    if (ptx::elect_one()) {
      // The thread that issues the loads needs about 390 cycles for a stage whatever its bytes (170 to look at the ring,
      // 215 to issue three loads), more than the MMAs of a narrow tile take: its stages hold two k-blocks each where the
      // ring has room (k_blocks_of_a_stage), which are loaded by as many loads as one.  One k-block a stage and two, us,
      // device: bf16 512 x 512 x 8192 16.0, 13.1; 4096 x 32 x 4096 9.1, 7.8.  Loops of their own: with the number of k-blocks
      // as a variable of one loop, products with one a stage were up to 15 % slower.
      // (Shared-memory and barrier addresses as plain integers, as few loads per stage as the boxes allow: the
      // thread that issues them is busy for about 100 cycles per load, which delays the refill of a stage.
      // Three loads instead of six (two m-blocks) or four: 49152 x 32 x 12288 bf16 123.1 -> 119.6 us, int8
      // 4096 x 8192 x 4096 79.3 -> 77.2, 256 x 256 x 512 4.55 -> 4.47.)
      int stage = 0;
      uint32_t phase = 0;
      constexpr int box_elems = C::kAtomElems;  // elements per 128-byte atom row
      const int b_atom = C::b_rows(tile_n) * kAtomBytes;
      const uint32_t ring = ptx::smem_u32(smem);
      const uint32_t full0 = CTAS == 2 ? ptx::map_to_cta(ptx::smem_u32(&sh->full[0]), 0) : ptx::smem_u32(&sh->full[0]);
      for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
        int mt, nt;
        tile_coords(t, p, mt, nt);
        // the last n-tile may be narrower: the pair then splits only the columns that exist
        const int n_eff = min(tile_n, (int)(p.N - (int64_t)nt * tile_n));
        const int col0 = nt * tile_n + (int)cta_rank * (n_eff / CTAS);  // first B row (N index)
        const int row0 = first_row<CTAS, MBLK>(mt, (int)cta_rank, (int)p.M);
        const uint32_t tx_bytes = (uint32_t)((C::kABytes + C::kEBytes + b_bytes) * CTAS);
        // implicit convolution: (image, row, column) of this CTA's first output pixel
        int conv_n = 0, conv_p = 0, conv_q = 0, conv_c0 = 0, conv_r = 0, conv_s = 0;
        if (p.conv) {
          conv_n = p.by_image(col0);
          const int rem = col0 - conv_n * p.conv_h * p.conv_w;
          conv_p = p.by_conv_w(rem);
          conv_q = rem - conv_p * p.conv_w;
        }
        // (Walking K backwards in every other tile of a CTA, so that a wave first meets the END of the A
        // panel the wave before it has just finished with, saves 12 % of the DRAM reads and 1.5 % of the
        // time, but makes the rounding of a result depend on which CTA computed its tile: the same rows
        // and columns would no longer give the same bits when M or N is split differently.  Not done.)
        if (kps == 2) {  // (A in whole 128-byte atoms: its atoms are a third dimension as B's are)
          for (int kb = 0; kb < p.k_blocks; kb += 2) {
            if (!bounded_wait(&sh->empty[stage], phase ^ 1u, sh, p.status, 1u, wait_limit())) break;
            if (!(p.test_skip_stage && t == cluster_id && kb == 2)) {  // (test hook: as below)
              const uint32_t sa = ring + stage * slot_bytes, sb = sa + 2 * C::kABytes, se = sb + 2 * b_bytes;
              const uint32_t full = full0 + 8 * stage;
              if (cta_rank == 0) ptx::mbar_expect_tx(&sh->full[stage], 2 * tx_bytes);
              ptx::tma_load_3d<CTAS>(se, &map_e, full, 0, 16 * kb * C::kEBlocks, row0 / kBlockM);
              ptx::tma_load_3d<CTAS>(sa, &map_a, full, 0, row0, kb);
              ptx::tma_load_3d<CTAS>(sb, &map_b, full, 0, col0, kb * C::kBBoxes);
            }
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
          }
          continue;
        }
        for (int kb = kb_begin; kb < kb_end; ++kb) {
          if (!bounded_wait(&sh->empty[stage], phase ^ 1u, sh, p.status, 1u, wait_limit())) break;
          if (p.test_skip_stage && (!SPLIT || p.test_skip_stage == 1 || p.test_skip_stage == 2 + split_rank) && t == cluster_id &&
              kb == kb_begin + 1) {
            // test hook: this k-block of the first tile is neither armed nor loaded by either CTA (by one of those that share
            // the tile's k-blocks), so the MMA issuer's wait for it expires and every role leaves through the abort path
            if (++stage == p.stages) { stage = 0; phase ^= 1u; }
            continue;
          }
          const uint32_t sa = ring + stage * slot_bytes, sb = sa + C::kABytes, se = sb + b_bytes;
          const uint32_t full = full0 + 8 * stage;
          if (cta_rank == 0) ptx::mbar_expect_tx(&sh->full[stage], tx_bytes);
          // both m-blocks' rows and metadata blocks are neighbours: one box each
          if (SPARSE) ptx::tma_load_3d<CTAS>(se, &map_e, full, 0, 16 * kb * C::kEBlocks, row0 / kBlockM);
#pragma unroll
          for (int i = 0; i < C::kABoxes; ++i)
            ptx::tma_load_2d<CTAS>(sa + i * MBLK * kBlockM * kAtomBytes, &map_a, full, (kb * C::kABoxes + i) * box_elems, row0);
          if (B_MN) {
            // B stored N-contiguous: boxes of 128 bytes along N x all k-rows of the stage
            for (int c = 0; c < C::b_chunks(tile_n); ++c)
              ptx::tma_load_2d<CTAS>(sb + c * C::kBChunkBytes, &map_b, full, col0 + c * C::kBChunkElems, kb * C::kKPerStage);
          } else if (p.conv) {
            // k = (r * 3 + s) * C + c: a stage holds channels of one filter tap; rows = output pixels
#pragma unroll
            for (int i = 0; i < C::kBBoxes; ++i)
              ptx::tma_load_im2col_4d<CTAS>(sb + i * b_atom, &map_b, full, conv_c0 + i * box_elems, conv_q - 1,
                                            conv_p - 1, conv_n, (uint16_t)conv_s, (uint16_t)conv_r);
            conv_c0 += C::kKPerStage;
            if (conv_c0 == p.conv_c) {
              conv_c0 = 0;
              if (++conv_s == 3) { conv_s = 0; ++conv_r; }
            }
          } else if (p.b_3d) {
            ptx::tma_load_3d<CTAS>(sb, &map_b, full, 0, col0, kb * C::kBBoxes);
          } else {
#pragma unroll
            for (int i = 0; i < C::kBBoxes; ++i)
              ptx::tma_load_2d<CTAS>(sb + i * b_atom, &map_b, full, (kb * C::kBBoxes + i) * box_elems, col0);
          }
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        }
      }
      // (teardown of a pair: the last commits, which come from CTA 0, have arrived)
      if (CTAS == 2 && !sh->abort)
        drain_ring(p.stages, stage, phase, [&](int s, uint32_t parity) {
          return bounded_wait(&sh->empty[s], parity, sh, p.status, 1u, wait_limit());
        });
    }
  } else if (warp == 1) {
    // ------------------------------ MMA issuer ------------------------------
    if (cta_rank == 0 && ptx::elect_one()) {
      const int b_atom = C::b_rows(tile_n) * kAtomBytes;
      const uint32_t ring = ptx::smem_u32(smem);
      int stage = 0, acc = 0;
      uint32_t phase = 0, acc_phase = 0, e_buf = 0;
      for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
        int mt, nt;
        tile_coords(t, p, mt, nt);
        // instruction N = the columns this tile really has (a multiple of 16, of 32 for int8)
        const int n_eff = min(tile_n, (int)(p.N - (int64_t)nt * tile_n));
        const int live = live_blocks<CTAS, MBLK>(mt, (int)p.M);  // m-blocks with rows (others are not multiplied)
        const uint32_t idesc = make_idesc<KIND>(SPARSE, B_MN, p.a_fmt, kBlockM * CTAS, n_eff, KIND == 0 && p.acc_f16);
        // the MMAs of a k-block: A, B and metadata at sa, sb, se
        auto multiply = [&](int kb, uint32_t sa, uint32_t sb, uint32_t se) {
          // metadata columns alternate between two small tensor-memory buffers from k-block to k-block
          const uint32_t e_base = tmem_base + C::kECol + e_buf * (MBLK * 8);
          e_buf ^= 1u;
          if (SPARSE) {
#pragma unroll
            for (int j = 0; j < MBLK; ++j) {
              if (j >= live) break;
#pragma unroll
              for (int i = 0; i < C::kEBlocks; ++i)
                ptx::tmem_cp_128x128b<CTAS>(e_base + j * 8 + 4 * i,
                                            ptx::smem_desc(se + j * C::kEBlockBytes + i * 2048, ptx::kLayoutNone, 128));
            }
          }
          const uint64_t db0 = B_MN ? ptx::smem_desc(sb, C::kBMnLayout, C::kBMnSbo, C::kBChunkBytes) : ptx::smem_desc(sb, ptx::kLayoutSw128, 1024);
#pragma unroll
          for (int j = 0; j < MBLK; ++j) {
            if (j >= live) break;
            const uint32_t d_tmem = tmem_base + (acc * MBLK + j) * BLOCK_N;
            const uint32_t e_tmem = e_base + j * 8;
            const uint64_t da0 = ptx::smem_desc(sa + j * C::kABlockBytes, ptx::kLayoutSw128, 1024);
#pragma unroll
            for (int k = 0; k < C::kMmasPerStage; ++k) {
              const uint32_t accumulate = (kb > 0 || k > 0) ? 1u : 0u;
              if (SPARSE) {
                // 32 bytes of compressed A and 64 bytes of B per instruction
                const uint64_t da = ptx::desc_at(da0, k * 32);
                const uint64_t db = ptx::desc_at(db0, B_MN ? k * C::kBKStepBytes : (k >> 1) * b_atom + (k & 1) * 64);
                if (!one_byte_operands(KIND)) {
                  // one 32-bit metadata column per instruction: even-aligned address + selector
                  ptx::mma_sparse<KIND, CTAS>(d_tmem, da, db, e_tmem + (k & ~1), idesc | (uint32_t)(k & 1), accumulate);
                } else {
                  ptx::mma_sparse<KIND, CTAS>(d_tmem, da, db, e_tmem + 2 * k, idesc, accumulate);
                }
              } else {
                const uint64_t da = ptx::desc_at(da0, (k >> 2) * kBlockM * kAtomBytes + (k & 3) * 32);
                const uint64_t db = ptx::desc_at(db0, B_MN ? k * C::kBKStepBytes : (k >> 2) * b_atom + (k & 3) * 32);
                ptx::mma_dense<KIND, CTAS>(d_tmem, da, db, idesc, accumulate);
              }
            }
          }
        };
        if (!bounded_wait(&sh->tmem_empty[acc], acc_phase ^ 1u, sh, p.status, 2u, wait_limit())) break;
        ptx::tc_fence_after();
        bool ok = true;
        // the stage may be refilled once its MMAs have read it
        auto release = [&] {
          if (CTAS == 1) ptx::tc_commit(&sh->empty[stage]);
          else ptx::tc_commit_pair(&sh->empty[stage], 3);
          if (++stage == p.stages) { stage = 0; phase ^= 1u; }
        };
        if (kps == 2) {
          for (int kb = 0; kb < p.k_blocks; kb += 2) {
            if (!bounded_wait(&sh->full[stage], phase, sh, p.status, 3u, wait_limit())) { ok = false; break; }
            ptx::tc_fence_after();
            const uint32_t sa = ring + stage * slot_bytes, sb = sa + 2 * C::kABytes, se = sb + 2 * b_bytes;
            multiply(kb, sa, sb, se);
            if (kb + 1 < p.k_blocks) multiply(kb + 1, sa + C::kABytes, sb + b_bytes, se + C::kEAlloc);
            release();
          }
        } else {
          for (int kb = kb_begin; kb < kb_end; ++kb) {
            if (!bounded_wait(&sh->full[stage], phase, sh, p.status, 3u, wait_limit())) { ok = false; break; }
            ptx::tc_fence_after();
            const uint32_t sa = ring + stage * slot_bytes;
            multiply(kb - kb_begin, sa, sa + C::kABytes, sa + C::kABytes + b_bytes);
            release();
          }
        }
        if (!ok) break;
        if (CTAS == 1) ptx::tc_commit(&sh->tmem_full[acc]);
        else ptx::tc_commit_pair(&sh->tmem_full[acc], 3);
        if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
      }
      // (teardown of a pair: the last accumulators have been handed back, CTA 1's warps' arrivals among them)
      if (CTAS == 2 && !sh->abort)
        drain_ring(C::kAccStages, acc, acc_phase, [&](int a, uint32_t parity) {
          return bounded_wait(&sh->tmem_empty[a], parity, sh, p.status, 2u, wait_limit());
        });
    }
  } else if (warp >= kFirstEpiWarp) {
    // ------------------------------ epilogue ------------------------------
    if constexpr (!C::staged_epilogue(CS, COLS)) {
      // loads and stores by the epilogue warps themselves
      if (SPLIT) ptx::cluster_wait();  // (the set-up's: the other CTAs' barriers are there)
      epilogue_direct<KIND, CS, COLS, HAS_C, BLOCK_N, CTAS, MBLK, C::kAccStages, WARPS, SPLIT>(p, sh, epi, tmem_base, (int)cta_rank, cluster_id,
                                                                          num_clusters, num_tiles, warp, lane, ptx::smem_u32(b_ring), split_rank);
      // (all that this warp sends is on its way: the cluster may leave when every warp has come so far)
      if (SPLIT) {
        __syncwarp();
        ptx::cluster_arrive_relaxed();
      }
    } else {
    // 4-byte row-major outputs when every epilogue warp can have a box buffer of its own.  The two warps
    // of a lane quarter own its 32 accumulator rows and take its 32 x 32 boxes in turn: TMA load of the C
    // box (if beta != 0) into a staging buffer one box ahead, tcgen05.ld of the accumulator columns,
    // convert in place, TMA store of the D box.  Boxes outside the matrix are clipped by the TMA.
    const int q = warp & 3;  // tensor-memory lane quarter this warp may read
    const int ew = warp - kFirstEpiWarp;  // epilogue warp 0..7: warps ew and ew + 4 share a lane quarter
    constexpr int buf_bytes = 4096, split = 2;
    const int first_it = ew >> 2;
    const int warp_bytes = p.epi_bytes / kEpiWarps;
    const int nbuf = min(2, warp_bytes / buf_bytes);  // staging buffers of this warp: 1 or 2
    // (the buffer of box seq + 1 is claimed, for its C or its result, at the end of box seq: with two buffers one
    // store may still be reading its own then)
    uint8_t* my_bufs = epi + ew * warp_bytes;
    const int subs = tile_n / 32, iters = MBLK * subs;

    // box `it` of the tile (mt, nt): first row / column and whether any of it lies inside the matrix
    auto box_of = [&](int mt, int nt, int it, int& row0, int& col0) -> bool {
      const int j = it >= subs, sc = it - j * subs;
      row0 = first_row<CTAS, MBLK>(mt, (int)cta_rank, (int)p.M) + j * kBlockM + q * 32;
      col0 = nt * tile_n + sc * 32;
      return j < live_blocks<CTAS, MBLK>(mt, (int)p.M) && row0 < p.M && col0 < p.N;
    };
    // cursor of the C loads over the same stream of boxes, one live box in front of the consumer
    // (the tile coordinates cost two divisions: once per tile, not per box)
    int pf_t = cluster_id, pf_it = first_it, pf_mt = 0, pf_nt = 0;
    if (pf_t < num_tiles) tile_coords(pf_t, p, pf_mt, pf_nt);
    uint32_t pf_seq = 0;
    auto issue_c_load = [&]() {  // lane 0 only: load the next live box of the stream, if any
      while (pf_t < num_tiles) {
        int row0, col0;
        const bool live_box = box_of(pf_mt, pf_nt, pf_it, row0, col0);
        pf_it += split;
        if (pf_it >= iters) {
          pf_it = first_it;
          pf_t += num_clusters;
          if (pf_t < num_tiles) tile_coords(pf_t, p, pf_mt, pf_nt);
        }
        if (live_box) {
          const int b = pf_seq % nbuf;
          ptx::mbar_expect_tx(&sh->c_full[ew][b], (uint32_t)buf_bytes);
          ptx::tma_load_2d<1>(ptx::smem_u32(my_bufs + b * buf_bytes), &map_c, ptx::smem_u32(&sh->c_full[ew][b]), col0, row0);
          ++pf_seq;
          return;
        }
      }
    };
    if (HAS_C && lane == 0) issue_c_load();

    int acc = 0;
    uint32_t acc_phase = 0, seq = 0;
    for (int t = cluster_id; t < num_tiles && !sh->abort; t += num_clusters) {
      int mt, nt;
      tile_coords(t, p, mt, nt);
      if (!bounded_wait(&sh->tmem_full[acc], acc_phase, sh, p.status, 4u, p.wait_limit)) break;
      ptx::tc_fence_after();
      uint32_t r_next[32];
      const uint32_t t_acc = tmem_base + (acc * MBLK) * BLOCK_N + ((uint32_t)(q * 32) << 16);
      // accumulator columns of box `it`
      auto acc_of = [&](int it) -> uint32_t { return t_acc + (it >= subs ? BLOCK_N + (it - subs) * 32 : it * 32); };
      if (first_it < iters) ptx::tmem_ld_32x32b(acc_of(first_it), r_next);  // (32 columns, one m-block: one box for two warps)
      bool ok = true;
#pragma unroll 1
      for (int it = first_it; it < iters; it += split) {
        uint32_t r[32];
        ptx::tmem_ld_wait(r_next);
#pragma unroll
        for (int e = 0; e < 32; ++e) r[e] = r_next[e];
        if (it + split < iters) ptx::tmem_ld_32x32b(acc_of(it + split), r_next);
        int row0, col0;
        if (!box_of(mt, nt, it, row0, col0)) continue;  // same answer for the whole warp
        const int b = seq % nbuf;
        uint8_t* buf = my_bufs + b * buf_bytes;
        if (HAS_C && !bounded_wait(&sh->c_full[ew][b], (seq / nbuf) & 1u, sh, p.status, 5u, p.wait_limit)) { ok = false; break; }
        if (KIND == 0 && p.acc_f16) widen_f16_accumulators(r);
        float scale = 1.f, bias = 0.f;
        if (KIND == 1 && p.dequant) {
          // this thread's output row: its scale and bias
          const int row = min(row0 + lane, (int)p.M - 1);
          scale = p.row_scale[row];
          bias = p.bias ? p.bias[row] : 0.f;
        }
        convert_row_staged<KIND, HAS_C>(r, buf, lane, p, scale, bias);
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) {
          ptx::tma_store_2d(&map_d, buf, col0, row0);
          ptx::bulk_commit_group();
          // the buffer claimed next is free once the store that used it last has read it
          if (nbuf == 2) ptx::bulk_wait_group_read<1>();
          else ptx::bulk_wait_group_read<0>();
          if (HAS_C) issue_c_load();
        }
        __syncwarp();
        ++seq;
      }
      if (!ok) break;
      // accumulators drained: hand them back to the MMA issuer (CTA 0 of the pair)
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) {
        if (CTAS == 1) ptx::mbar_arrive(&sh->tmem_empty[acc]);
        else ptx::mbar_arrive_cluster(&sh->tmem_empty[acc], 0);
      }
      if (++acc == C::kAccStages) { acc = 0; acc_phase ^= 1u; }
    }
    if (lane == 0) ptx::bulk_wait_group_read<0>();  // staging buffers must outlive the stores that read them
    }
  }

  // ------------------------------ teardown ------------------------------
  if (SPLIT && warp < kFirstEpiWarp) {
    __syncwarp();
    ptx::cluster_wait();
    ptx::cluster_arrive_relaxed();
  }
  ptx::tc_fence_before();
  __syncthreads();
  // after waits that were given up: copies issued before them, and the other CTA's arrivals, may still be landing in this
  // CTA's shared memory
  auto settle = [&] {
    if (sh->abort)
      for (int i = 0; i < 64; ++i) __nanosleep(1000);
  };
  settle();
  if (CTAS == 2) {
    // The pair leaves together.  The arrival orders no memory accesses, and need not: whatever a CTA sends to the other's
    // barriers has a waiter there (loads: the issuer; commits and hand-backs: later tiles and, for the last ones,
    // drain_ring above), and tensor memory has been read once tcgen05.wait::ld returns.  (With release instead of the issuer's
    // drain it also waits for D's stores: BERT FFN 12.4 against 12.1 us, device; large products the same.)
    ptx::cluster_arrive_relaxed();
    ptx::cluster_wait();
  } else if (SPLIT) {
    ptx::cluster_wait();  // (what was sent to this CTA has a waiter, split_full; after waits that were given up, settle() is it)
  }
  if (warp == 1) {
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc<CTAS>(tmem_base, kTmemCols);
  }
  if (CTAS == 2 || SPLIT) settle();
}

template <int KIND, bool SPARSE, int BLOCK_N, int CTAS, int MBLK, bool B_MN>
sp24_status launch(const TileShape& tile, const sp24_gemm_desc* d, const GemmParams& base, const void* A, const void* meta, const void* B,
                   cudaStream_t stream) {
  using C = Cfg<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN>;
  GemmParams p = base;
  const int tile_n = p.tile_n = tile.tile_n;
  p.split_log = can_split<KIND, SPARSE, CTAS, MBLK, B_MN> ? tile.split_log : 0;
  const int cs = elem_bytes(d->cd_type);
  // Shared-memory split.  The ring comes first (these kernels are bound by the operand feed: one
  // stage less cost the int8 configuration 9 %); a staged epilogue gets what is left.
  constexpr bool kTwelve = twelve_warps<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN>;
  int tile_m = kBlockM * CTAS * MBLK;
  const int warps = epilogue_warps<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN>(d, tile_n);
  p.epi_bytes = warps * (C::staged_epilogue(cs, p.cd_col_major) ? 4096 : 2048);
  const int es = KIND == 0 ? 2 : (one_byte_operands(KIND) ? 1 : 4);
  const uint32_t atom_elems = kAtomBytes / es;
  const uint64_t a_cols = SPARSE ? d->K / 2 : d->K;
  p.kps = p.split_log ? 1 : C::k_blocks_of_a_stage(tile_n, p.epi_bytes, (int64_t)a_cols, p.conv != 0);
  if (p.split_log) {  // (as epilogue_direct lays them out)
    const int cols = cs == 4 ? 16 : 32;
    p.part_bytes = ((1 << p.split_log) - 1) * (kEpiWarps >> p.split_log) * ((tile_n / cols + 1) / 2) * cols * 128;
  }
  int ring_bytes = C::stage_bytes(tile_n) * p.kps;
  p.stages = C::ring_stages(ring_bytes, p.epi_bytes + p.part_bytes);
  if constexpr (is_tall<CTAS, MBLK>) {
    tile_m = p.mblk * kBlockM;
    // slots of A (each k-block needs mblk) and of B: the split with the most of A in flight
    const int b_slot = C::b_bytes(tile_n), budget = C::kSmemLimit - p.epi_bytes;
    ring_bytes = C::kABlockBytes + C::kEBlockBytes;
    p.stages = 0;
    for (int bs = 2; bs <= 8 && bs * b_slot < budget; ++bs) {
      int slots = (budget - bs * b_slot) / ring_bytes;
      if (slots > (bs - 1) * p.mblk + 1) slots = (bs - 1) * p.mblk + 1;
      if (slots > C::kMaxStages) slots = C::kMaxStages;
      if (slots > p.stages) { p.stages = slots; p.b_stages = bs; }
    }
  }
  const uint32_t b_box_rows = (uint32_t)C::b_rows(tile_n);
  p.m_tiles = (int)((d->M + tile_m - 1) / tile_m);
  p.n_tiles = (int)((d->N + tile_n - 1) / tile_n);
  p.k_blocks = (int)((d->K + C::kKPerStage - 1) / C::kKPerStage);
  if (p.band > p.m_tiles) p.band = p.m_tiles;
  p.by_band_tiles = FastDiv::by((uint32_t)(p.band * p.n_tiles));
  p.by_band = FastDiv::by((uint32_t)p.band);
  p.by_last_band = FastDiv::by((uint32_t)((p.m_tiles - 1) % p.band + 1));
  // metadata blocks per 128-row block: 128 columns each (64 for the 1:2 pattern), an even number of them
  p.meta_kb = KIND == 2 ? (int)(2 * ((d->K + 127) / 128)) : (int)(2 * ((d->K + 255) / 256));
  CUtensorMap map_a, map_b, map_e;
  sp24_status st;
  if (p.kps == 2)
    st = make_map(&map_a, MapShape{A, {atom_elems, (uint64_t)d->M, a_cols / atom_elems}, {(uint64_t)d->lda * es, kAtomBytes},
                                   {atom_elems, kBlockM, 2}, es, 128});
  else
    st = make_map(&map_a, A, es, d->M, a_cols, d->lda * es, atom_elems, (is_tall<CTAS, MBLK> ? 1 : MBLK) * kBlockM, 128);
  if (st != SP24_OK) return st;
  if (p.conv) {
    // B = im2col view of the NHWC activation: boxes of b_rows output pixels x one 128-byte run of channels
    if (B_MN) return SP24_ERR_UNSUPPORTED;
    if (KIND == 2) return SP24_ERR_UNSUPPORTED;
    const uint64_t nb = (uint64_t)d->N / ((uint64_t)p.conv_h * p.conv_w);
    st = make_im2col_map(&map_b, B, es, nb, p.conv_h, p.conv_w, p.conv_c, atom_elems, b_box_rows);
  } else if (B_MN) {
    st = make_map(&map_b, B, es, d->K, d->N, d->ldb * es, C::kBChunkElems, C::kKPerStage,
                  KIND == 2 ? kSwizzle128Atom32 : 128);
  } else if (C::kBBoxes > 1 && d->K % atom_elems == 0) {
    // K in whole 128-byte atoms: the atoms of a stage are a third dimension, one load brings them all (a K tail
    // needs the zeros that only the two-dimensional map gives it)
    p.b_3d = 1;
    st = make_map(&map_b, MapShape{B, {atom_elems, (uint64_t)d->N, (uint64_t)d->K / atom_elems},
                                   {(uint64_t)d->ldb * es, kAtomBytes}, {atom_elems, b_box_rows, (uint32_t)(C::kBBoxes * p.kps)}, es, 128});
  } else {
    st = make_map(&map_b, B, es, d->N, d->K, d->ldb * es, atom_elems, b_box_rows, 128);
  }
  if (st != SP24_OK) return st;
  if (SPARSE) {
    // metadata as rows of 128 bytes: 16 * meta_kb of them per 128 rows of A
    st = make_map(&map_e, MapShape{meta, {128, (uint64_t)p.meta_kb * 16, (uint64_t)((d->M + 127) / 128)},
                                   {128, (uint64_t)p.meta_kb * 2048}, {128, (uint32_t)(16 * C::kEBlocks * p.kps), is_tall<CTAS, MBLK> ? 1 : MBLK}, 1, 0});
    if (st != SP24_OK) return st;
  } else {
    map_e = map_a;
  }
  CUtensorMap map_c, map_d;
  if (!C::staged_epilogue(cs, p.cd_col_major)) {
    map_c = map_d = map_a;  // not used
  } else {
    if (C::kSmemLimit - p.stages * ring_bytes >= 2 * p.epi_bytes) p.epi_bytes *= 2;
    // C and D move in 32 x 32 boxes whose rows are 128 bytes
    st = make_map(&map_d, p.D, cs, d->M, d->N, d->ldd * cs, 32, 32, 128);
    if (st != SP24_OK) return st;
    map_c = map_d;
    if (p.has_c) st = make_map(&map_c, p.C, cs, d->M, d->N, d->ldc * cs, 32, 32, 128);
    if (st != SP24_OK) return st;
  }
  // the kernels of the output forms
  using Kernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, CUtensorMap, GemmParams);
  constexpr bool kCanSplit = can_split<KIND, SPARSE, CTAS, MBLK, B_MN>;
  Kernel forms[24] = {}, twelve[2] = {};  // [split][with C][bytes][order]
#define SP24_FORM(CS_, COLS_, C_)                                                                                                   \
  forms[6 * C_ + 2 * (CS_ >> 1) + COLS_] = gemm_kernel<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN, CS_, COLS_, C_>;                     \
  if constexpr (kTwelve && CS_ == 1) twelve[COLS_] = gemm_kernel<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN, CS_, COLS_, false, false, 12>; \
  if constexpr (kCanSplit) forms[12 + 6 * C_ + 2 * (CS_ >> 1) + COLS_] = gemm_kernel<KIND, SPARSE, BLOCK_N, CTAS, MBLK, B_MN, CS_, COLS_, C_, true>;
  if constexpr (KIND == 1) { SP24_FORM(1, false, false) SP24_FORM(1, true, false) }
  if constexpr (KIND != 2) { SP24_FORM(2, false, false) SP24_FORM(2, true, false) }
  if constexpr (KIND != 2 && KIND != 1) { SP24_FORM(2, false, true) SP24_FORM(2, true, true) }  // (int8: only INT32 results are added to)
  if constexpr (BLOCK_N % 32 == 0) {  // 240-column tiles: 2-byte outputs only
    SP24_FORM(4, false, false) SP24_FORM(4, true, false) SP24_FORM(4, false, true) SP24_FORM(4, true, true)
  }
#undef SP24_FORM
  const Kernel kernel = warps == 12 ? twelve[p.cd_col_major] : forms[12 * (p.split_log != 0) + 6 * p.has_c + 2 * (cs >> 1) + p.cd_col_major];
  if (kernel == nullptr) return SP24_ERR_UNSUPPORTED;
  {
    // the shared-memory opt-in is per kernel and device: once is enough (by several threads at a time does no harm).  All
    // forms at once, so that a call with one form also loads the others' code: none is loaded for the first time inside a
    // stream capture after that.
    static std::atomic<bool> done[64];
    int dev = 0;
    SP24_CUDA_CHECK(cudaGetDevice(&dev));
    const bool kept = dev >= 0 && dev < 64;
    if (!kept || !done[dev].load(std::memory_order_acquire)) {
      for (int i = 0; i < 26; ++i)
        if (const Kernel k = i < 24 ? forms[i] : twelve[i - 24]) SP24_CUDA_CHECK(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, C::kSmemBytes));
      if (kept) done[dev].store(true, std::memory_order_release);
    }
  }
  const int tiles = p.m_tiles * p.n_tiles;
  int clusters = sm_count() / CTAS;
  if (clusters > tiles || p.split_log) clusters = tiles;  // (k-blocks shared: one tile to a cluster)
  const int cluster_ctas = CTAS << p.split_log;
  return launch_overlapped(kernel, dim3((unsigned)(clusters * cluster_ctas)), dim3(32 * (kFirstEpiWarp + warps)), C::kSmemBytes, stream, cluster_ctas, map_a,
                           map_b, map_e, map_c, map_d, p);
}

}  // namespace

template <int KIND>
sp24_status launch_gemm(TileShape t, bool sparse, bool b_mn, const sp24_gemm_desc* d, const GemmParams& p, const void* A,
                        const void* meta, const void* B, cudaStream_t s) {
  constexpr bool tf32 = KIND == 2;
  auto is = [&](int ctas, int block_n, int mblk) { return t.ctas == ctas && t.block_n == block_n && t.mblk == mblk; };
#define SP24_SHAPE(CT, BN, MB, MN)                                     \
  if (is(CT, BN, MB) && b_mn == MN)                                    \
    return sparse ? launch<KIND, true, BN, CT, MB, MN>(t, d, p, A, meta, B, s) : launch<KIND, false, BN, CT, MB, MN>(t, d, p, A, meta, B, s);
  SP24_SHAPE(1, 128, 1, false)
  SP24_SHAPE(2, 224, 1, false)
  SP24_SHAPE(2, 224, 2, false)
  SP24_SHAPE(2, 256, 1, false)
  SP24_SHAPE(1, 128, 1, true)
  SP24_SHAPE(2, 224, 1, true)
  SP24_SHAPE(2, 224, 2, true)
  if constexpr (KIND == 0 || KIND == 1) {
    SP24_SHAPE(2, 192, 2, false)
  }
  if constexpr (KIND == 0) {
    SP24_SHAPE(2, 240, 1, false)  // 2-byte outputs only
  }
  if constexpr (!tf32)  // dense variant only
    if (is(2, 256, 2) && !sparse && !b_mn) return launch<KIND, false, 256, 2, 2, false>(t, d, p, A, meta, B, s);
  if (t.ctas == 1 && t.block_n == 128 && (t.mblk == 2 || t.mblk == kTallBlocks) && sparse && !b_mn)
    return launch<KIND, true, 128, 1, kTallBlocks, false>(t, d, p, A, meta, B, s);
#undef SP24_SHAPE
  return SP24_ERR_UNSUPPORTED;
}

}  // namespace sp24
