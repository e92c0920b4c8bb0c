// Streaming kernels of the 2:4 path: magnitude pruning (Section 4.1 step 2), compression to
// kept values + 2-bit position metadata and its inverse (Section 3.1, Figure 1), and the
// im2col lowering of a 3x3 convolution (Section 4.2).  All of them are bound by HBM bandwidth:
// every thread moves whole 16-byte vectors, the selection is a handful of integer compares.
#include "sp24_common.cuh"

namespace sp24 {
namespace {

// ---- selection -------------------------------------------------------------------------
// Bit p of the result is set iff position p of the group is kept.  Position a beats position b
// (a < b) when key[a] >= key[b] -- equal magnitudes go to the lower index -- so the six
// comparisons define a strict total order and exactly two positions are beaten fewer than
// two times.
__device__ __forceinline__ uint32_t keep_mask4(uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3) {
  uint32_t c01 = k0 >= k1, c02 = k0 >= k2, c03 = k0 >= k3;
  uint32_t c12 = k1 >= k2, c13 = k1 >= k3, c23 = k2 >= k3;
  uint32_t b0 = 3u - (c01 + c02 + c03);
  uint32_t b1 = c01 + 2u - (c12 + c13);
  uint32_t b2 = c02 + c12 + 1u - c23;
  uint32_t b3 = c03 + c13 + c23;
  return (b0 < 2u) | ((b1 < 2u) << 1) | ((b2 < 2u) << 2) | ((b3 < 2u) << 3);
}

// keep mask (two bits set) -> metadata nibble p0 | p1 << 2.
__device__ __forceinline__ uint32_t mask_to_nibble(uint32_t mask) {
  uint32_t p0 = __ffs(mask) - 1, p1 = 31 - __clz(mask);
  return p0 | (p1 << 2);
}

// Magnitude key of an 8-bit element: |x| for int8 (-128 -> 0x80 = 128, no saturation), the seven
// bits below the sign for the 8-bit floating-point types (`f8` != 0).
__device__ __forceinline__ uint32_t key8(uint32_t e, int f8) { return f8 ? (e & 0x7Fu) : (uint32_t)abs((int)(int8_t)e); }

// ---- prune -----------------------------------------------------------------------------
// Any alignment / leading dimension: one thread per group, element-wise accesses.
template <typename T>
__global__ void prune_scalar_kernel(const T* __restrict__ x, int64_t ldx, T* y, int64_t ldy, int64_t groups_per_row,
                                    int64_t total, int f8) {
  int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= total) return;
  int64_t row = id / groups_per_row, g = id - row * groups_per_row;
  const T* src = x + row * ldx + 4 * g;
  T e[4];
  uint32_t key[4];
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    e[p] = src[p];
    key[p] = sizeof(T) == 2 ? (uint32_t)((uint16_t)e[p] & 0x7FFFu) : key8((uint32_t)(uint8_t)e[p], f8);
  }
  uint32_t m = keep_mask4(key[0], key[1], key[2], key[3]);
  T* dst = y + row * ldy + 4 * g;
#pragma unroll
  for (int p = 0; p < 4; ++p) dst[p] = (m >> p) & 1u ? e[p] : (T)0;
}

// ---- metadata addressing ------------------------------------------------------------------
// Byte offset of the 16 metadata bits of chunk `chunk` (16 consecutive columns of A = four
// groups) of row `row`.  Canonical: K/8 bytes per row.  Operand order: 2048-byte blocks of 128
// rows x 128 columns, block (mb, kb) at (mb * KB + kb) * 2048.  Inside a block a 16-bit-type row
// r shares 32-bit words with row r+8 of its 16-row band, the second 16-column half of every
// 32-column slice lives 128 bytes further on, and each 32-column slice is one 32-bit tensor-
// memory column; an int8 row is simply 16 consecutive bytes.
template <int ES>
__device__ __forceinline__ int64_t meta_offset(int layout, int64_t row, int64_t chunk, int64_t K, int64_t KB) {
  if (layout == SP24_META_CANONICAL) return row * (K >> 3) + 2 * chunk;
  int64_t blk = (row >> 7) * KB + (chunk >> 3);
  int r = (int)(row & 127), cl = (int)(chunk & 7);
  int in_blk = ES == 2 ? 16 * (r & 7) + 2 * ((r >> 3) & 1) + 256 * (r >> 4) + 128 * (cl & 1) + 4 * (cl >> 1)
                       : 16 * r + 2 * cl;
  return blk * 2048 + in_blk;
}

// ---- selection of the vector kernels ------------------------------------------------------
// A 16-byte vector is transposed so that word i holds element i of all its groups (two in 16-bit lanes, four in 8-bit
// ones): each of the six comparisons is then one subtraction for all groups, whose result is the lane's top bit, and what
// follows is logic on those bits.  No table: with one in shared memory, indexed by the six bits, a vector took 88
// instructions and the look-ups met in the banks; it took 57 (ALU pipe 73 % busy) with the kept values gathered by lane masks and
// takes 53 (50 %) now that the bits are turned into byte-permute selectors by dot products, which run beside the ALU pipe.
__device__ __forceinline__ uint32_t prmt(uint32_t a, uint32_t b, uint32_t sel) {  // __byte_perm with the selectors that copy a sign
  uint32_t d;
  asm("prmt.b32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(sel));
  return d;
}

template <int ES>
__device__ __forceinline__ void transpose(uint4 w, uint32_t (&p)[4]) {
  if constexpr (ES == 2) {
    p[0] = prmt(w.x, w.z, 0x5410); p[1] = prmt(w.x, w.z, 0x7632); p[2] = prmt(w.y, w.w, 0x5410); p[3] = prmt(w.y, w.w, 0x7632);
  } else {
    const uint32_t t0 = prmt(w.x, w.y, 0x5140), t1 = prmt(w.z, w.w, 0x5140), t2 = prmt(w.x, w.y, 0x7362), t3 = prmt(w.z, w.w, 0x7362);
    p[0] = prmt(t0, t1, 0x5410); p[1] = prmt(t0, t1, 0x7632); p[2] = prmt(t2, t3, 0x5410); p[3] = prmt(t2, t3, 0x7632);
  }
}
template <int ES>
__device__ __forceinline__ uint4 transpose_back(const uint32_t (&p)[4]) {
  if constexpr (ES == 2)
    return make_uint4(prmt(p[0], p[1], 0x5410), prmt(p[2], p[3], 0x5410), prmt(p[0], p[1], 0x7632), prmt(p[2], p[3], 0x7632));
  const uint32_t a = prmt(p[0], p[1], 0x5140), b = prmt(p[2], p[3], 0x5140), c = prmt(p[0], p[1], 0x7362), d = prmt(p[2], p[3], 0x7362);
  return make_uint4(prmt(a, b, 0x5410), prmt(a, b, 0x7632), prmt(c, d, 0x5410), prmt(c, d, 0x7632));
}

// The selection of a transposed vector.  (Top bit of each lane; the others are not defined.)
template <int ES>
struct Selection {
  static constexpr uint32_t kTop = ES == 2 ? 0x80008000u : 0x80808080u;
  uint32_t key[4];   // magnitudes (16-bit types: below the top bit; 8-bit types: 0..128)
  uint32_t kept[4];  // is position i kept
  // Position 0 is kept if it beats two of the others, and so on (see keep_mask4).
  static __device__ __forceinline__ uint32_t majority(uint32_t a, uint32_t b, uint32_t c) { return (a & b) | (a & c) | (b & c); }
  // a >= b: with a's top bit set no lane borrows from the next.  8-bit keys use the top bit themselves (int8 -128): it
  // decides, and if equal the rest does.
  static __device__ __forceinline__ uint32_t at_least(uint32_t a, uint32_t b) {
    if constexpr (ES == 2) return (a | kTop) - b;
    const uint32_t rest = (a | kTop) - (b & ~kTop);
    return (a & ~b) | (~(a ^ b) & rest);
  }
  __device__ __forceinline__ Selection(const uint32_t (&p)[4], int f8) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (ES == 2) {
        key[i] = p[i] & ~kTop;
      } else {
        const uint32_t sign = prmt(p[i], 0, 0xBA98);
        key[i] = f8 ? p[i] & ~kTop : (p[i] ^ sign) + (sign & 0x01010101u);
      }
    }
    const uint32_t c01 = at_least(key[0], key[1]), c02 = at_least(key[0], key[2]), c03 = at_least(key[0], key[3]);
    const uint32_t c12 = at_least(key[1], key[2]), c13 = at_least(key[1], key[3]), c23 = at_least(key[2], key[3]);
    kept[0] = majority(c01, c02, c03);
    kept[1] = majority(~c01, c12, c13);
    kept[2] = majority(~c02, ~c12, c23);
    kept[3] = majority(~c03, ~c13, ~c23);
  }
  // Bit i of the metadata nibble: first kept position in bits 0 and 1, second in bits 2 and 3.
  template <int I>
  __device__ __forceinline__ uint32_t nibble_bit() const {
    return I == 0 ? ~kept[0] & kept[1] : I == 1 ? ~(kept[0] | kept[1]) : I == 2 ? kept[3] | ~kept[2] : kept[3] | kept[2];
  }
  __device__ __forceinline__ uint32_t keep_mask(int i) const { return prmt(kept[i], 0, ES == 2 ? 0xBB99u : 0xBA98u); }
  // The vector with the positions that are not kept set to zero.
  __device__ __forceinline__ uint4 pruned(const uint32_t (&p)[4]) const {
    const uint32_t y[4] = {p[0] & keep_mask(0), p[1] & keep_mask(1), p[2] & keep_mask(2), p[3] & keep_mask(3)};
    return transpose_back<ES>(y);
  }
  // Non-zero magnitudes that are not kept.
  __device__ __forceinline__ uint32_t lost() const {
    uint32_t n = 0;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t d = key[i] & ~keep_mask(i);
      n += __popc((((d & ~kTop) + ~kTop) | d) & kTop);
    }
    return n;
  }
};

// c + the sum of weights[i] over the bytes of `bits` that are 0xFF (the others are 0).  The weights are given as the bytes of
// their negatives, because such a byte counts as -1.
__device__ __forceinline__ uint32_t weigh(uint32_t bits, uint32_t minus_weights, uint32_t c) {
  return (uint32_t)__dp4a((int)bits, (int)minus_weights, (int)c);
}

// The kept values of a vector (8 bytes) and its metadata: two groups of a 16-bit type (8 bits), four of an 8-bit type (16).
template <int ES>
__device__ __forceinline__ uint32_t gather_kept(const Selection<ES>& s, uint4 w, uint32_t (&kept)[2]) {
  const uint32_t bit0 = s.template nibble_bit<0>(), bit1 = s.template nibble_bit<1>(), bit2 = s.template nibble_bit<2>(), bit3 = s.template nibble_bit<3>();
  if constexpr (ES == 2) {
    // bytes: bit 0 and bit 1 of group 0, of group 1; bits 2 and 3 likewise
    const uint32_t b01 = prmt(bit0, bit1, 0xFBD9), b23 = prmt(bit2, bit3, 0xFBD9);
    // a kept position i takes bytes 2i and 2i + 1 of the group's two words: selector nibbles 0x10 + 0x22 * i
    kept[0] = prmt(w.x, w.y, 256 * weigh(b23, 0x0000BCDEu, 0) + weigh(b01, 0x0000BCDEu, 0x1010));
    kept[1] = prmt(w.z, w.w, 256 * weigh(b23, 0xBCDE0000u, 0) + weigh(b01, 0xBCDE0000u, 0x1010));
    return weigh(b01, 0xE0F0FEFFu, weigh(b23, 0x80C0F8FCu, 0));  // 1, 2, 16, 32 and 4, 8, 64, 128
  } else {
    uint32_t meta[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {  // groups 0 and 1, groups 2 and 3: two words of one permutation
      const uint32_t b01 = prmt(bit0, bit1, h ? 0xFBEAu : 0xD9C8u), b23 = prmt(bit2, bit3, h ? 0xFBEAu : 0xD9C8u);
      const uint32_t first = weigh(b01, 0x0000FEFFu, weigh(b23, 0x0000E0F0u, 0x4400)), second = weigh(b01, 0xFEFF0000u, weigh(b23, 0xE0F00000u, 0));
      kept[h] = prmt(h ? w.z : w.x, h ? w.w : w.y, 256 * second + first);
      meta[h] = weigh(b01, 0xE0F0FEFFu, weigh(b23, 0x80C0F8FCu, 0));
    }
    return 256 * meta[1] + meta[0];
  }
}

// ---- prune (vectorised) -------------------------------------------------------------------------
// Launch geometry: blockDim = (TX, 256/TX), a warp always lies inside one row; thread (tx, ty) of block (bx, by) handles
// vectors (bx*UNROLL + u)*TX + tx, u < UNROLL, of rows by*TY + ty, + gridDim.y*TY, ...  No integer division on the device.
// One 16-byte vector per thread and unroll step; `vpr` vectors per row.  HBM-bound (6.5
// TB/s); us, device, with a table of selectors and now: int8 12288 x 3072 20.3, 13.8, 49152 x 12288 269, 184; bf16 the same.
template <int ES, int UNROLL>
__global__ void __launch_bounds__(kThreads) prune_vec_kernel(const uint8_t* x, int64_t row_bytes_x,
                                                             uint8_t* y, int64_t row_bytes_y, int64_t vpr,
                                                             int64_t rows, int f8) {
  wait_for_stream();
  const uint32_t c0 = blockIdx.x * UNROLL * blockDim.x + threadIdx.x;
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < rows;
       row += (int64_t)gridDim.y * blockDim.y) {
    const uint8_t* xr = x + row * row_bytes_x;
    uint8_t* yr = y + row * row_bytes_y;
    uint4 v[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t c = c0 + u * blockDim.x;
      if (c < vpr) v[u] = ld_stream(xr + c * 16u);
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t c = c0 + u * blockDim.x;
      if (c < vpr) {
        uint32_t p[4];
        transpose<ES>(v[u], p);
        st_stream(yr + c * 16u, Selection<ES>(p, f8).pruned(p));
      }
    }
  }
}

// ---- compress (fused prune + compress) ----------------------------------------------------
template <bool COUNT>
__device__ __forceinline__ void count_dropped(uint32_t lost, unsigned long long* dropped) {
  if (!COUNT) return;
  lost = __reduce_add_sync(0xFFFFFFFFu, lost);
  __shared__ uint32_t warp_sum[kThreads / 32];
  const int t = threadIdx.x;
  if ((t & 31) == 0) warp_sum[t >> 5] = lost;
  __syncthreads();
  if (t == 0) {
    uint32_t s = 0;
#pragma unroll
    for (int wi = 0; wi < kThreads / 32; ++wi) s += warp_sum[wi];
    if (s) atomicAdd(dropped, (unsigned long long)s);
  }
}

// Work unit ("cell"): 32 bytes of a row (16 columns of a 16-bit type, 32 of an 8-bit one) = 16 bytes of values and 2 or 4
// bytes of metadata.  A thread has a cell of the rows r and r + 8 of a 16-row group: in the operand order of a 16-bit type the
// two share each 32-bit word.  A warp has 16 cells of 2 neighbouring rows (8 of 4 rows where the row ends in half of that) and
// their partners, so that it writes whole 32-byte sectors of metadata: with 16-byte units and a row to a warp
// metadata went out in 2-byte pieces.  gridDim.y strides over the row groups.
// The domain is padded (rows to a multiple of 128, columns of 256) so that the operand order gets its 0x4 padding nibbles from
// the same launch.  HW: metadata straight into that order.  FULL: the launch covers exactly the matrix, so no bounds are
// checked.  PRUNE: the pruned matrix is written as well (y, same shape as x; may be x itself), so that one pass over x yields
// everything the separate prune and compress passes would.
// Bound by HBM where the matrix is large and cold.  Where it comes out of the L2 (bf16 12288 x 3072 right after apply_mask: 5 of
// 75 MB read from DRAM) the longest stall is memory and the ALU pipe half busy (52 %, 53 instructions a vector).  Us, device, table
// kernels of before / now: compress bf16 49152 x 12288 332, 281 (6.7 TB/s); 4096 x 4096 9.0, 7.4; 49152 x 256 13.4, 5.9; int8
// 49152 x 12288 292, 160; 12288 x 3072 22.0, 11.1; fused with prune bf16 49152 x 12288 534, 474; int8 340, 247; after
// apply_mask, both calls, bf16 12288 x 3072 40.4, 36.0.
// (Registers: five blocks an SM where nothing spills; 8-bit types are faster with four.)
template <int ES, bool COUNT, bool PRUNE>
constexpr int kCompressBlocks = ES == 2 && !COUNT && !PRUNE ? 5 : 4;

template <bool COUNT, bool PRUNE>
constexpr int kUnitBlocks = COUNT && PRUNE ? 4 : 5;

template <int ES, bool COUNT, bool HW, bool FULL, bool PRUNE>
__global__ void __launch_bounds__(kThreads, kCompressBlocks<ES, COUNT, PRUNE>)
compress_kernel(const uint8_t* x, int64_t row_bytes_x, uint8_t* vals, int64_t row_bytes_v, uint8_t* meta, int64_t M, int64_t K,
                uint32_t row_groups, uint32_t cells_pad, int cell_shift, int wide, unsigned long long* dropped, int f8, uint8_t* y,
                int64_t row_bytes_y) {
  constexpr uint32_t kCols = ES == 2 ? 16 : 32;  // columns of a cell
  wait_for_stream();
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t rows_of_warp = 32u >> cell_shift, cell = (blockIdx.x << cell_shift) + (lane & ((1u << cell_shift) - 1u));
  const uint32_t thread_row = warp * rows_of_warp + (lane >> cell_shift);  // eight of these to a row group
  const uint32_t in_group = thread_row & 7u, step = gridDim.y * rows_of_warp;
  const bool live_cell = FULL || (int64_t)cell * kCols < K, meta_cell = FULL || cell < cells_pad;
  const bool half_cell = ES == 1 && !FULL && K - (int64_t)cell * kCols == 16;
  // metadata of the cell in the first row of its 128-row block that this thread may have (canonical: in row 0)
  const uint32_t chunk = ES == 2 ? cell : 2 * cell, KB = ES == 2 ? cells_pad >> 3 : cells_pad >> 2;
  uint8_t* const meta_cell0 = meta + (!HW ? 2 * chunk
                                          : (chunk >> 3) * 2048u + 16u * in_group +
                                                (ES == 2 ? 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) : 2u * (chunk & 7u)));
  uint32_t n = blockIdx.y * rows_of_warp + (thread_row >> 3);  // row group
  const int64_t row0 = (int64_t)n * 16 + in_group;
  const uint8_t* xp = x + row0 * row_bytes_x + (int64_t)cell * 32;
  uint8_t* vp = vals + row0 * row_bytes_v + (int64_t)cell * 16;
  uint8_t* yp = PRUNE ? y + row0 * row_bytes_y + (int64_t)cell * 32 : nullptr;
  uint32_t lost = 0;
#pragma unroll 1
  for (; n < row_groups; n += step, xp += (int64_t)step * 16 * row_bytes_x, vp += (int64_t)step * 16 * row_bytes_v) {
    uint4 in[2][2];
    bool live[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      live[h] = live_cell && (FULL || (int64_t)n * 16 + in_group + 8 * h < M);
      if (live[h]) {
        const uint8_t* src = xp + 8 * h * row_bytes_x;
        if (wide & kWideX) {
          ld_stream32(src, in[h]);
        } else {
          in[h][0] = ld_stream(src);
          in[h][1] = half_cell ? make_uint4(0, 0, 0, 0) : ld_stream(src + 16);
        }
      }
    }
    uint32_t bits[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bits[h] = ES == 2 ? 0x4444u : 0x44444444u;  // padding: positions (0, 1) in all groups
      if (live[h]) {
        uint32_t kept[2][2], m[2];
        uint4 out[2];
#pragma unroll
        for (int v = 0; v < 2; ++v) {
          uint32_t p[4];
          transpose<ES>(in[h][v], p);
          const Selection<ES> s(p, f8);
          m[v] = gather_kept<ES>(s, in[h][v], kept[v]);
          if (PRUNE) out[v] = s.pruned(p);
          if (COUNT) lost += s.lost();
        }
        bits[h] = m[1] * (ES == 2 ? 256u : 65536u) + m[0];
        uint8_t* v = vp + 8 * h * row_bytes_v;
        if (ES == 2 || (wide & kWideVals)) {
          st_stream(v, make_uint4(kept[0][0], kept[0][1], kept[1][0], kept[1][1]));
        } else {
          __stcs(reinterpret_cast<uint2*>(v), make_uint2(kept[0][0], kept[0][1]));
          if (!half_cell) __stcs(reinterpret_cast<uint2*>(v + 8), make_uint2(kept[1][0], kept[1][1]));
        }
        if (PRUNE) {
          uint8_t* dst = yp + 8 * h * row_bytes_y;
          if (wide & kWideY) {
            st_stream32(dst, out);
          } else {
            st_stream(dst, out[0]);
            if (!half_cell) st_stream(dst + 16, out[1]);
          }
        }
      }
    }
    if (PRUNE) yp += (int64_t)step * 16 * row_bytes_y;
    if (!meta_cell) continue;
    if constexpr (HW) {
      uint8_t* mr = meta_cell0 + ((uint64_t)(n >> 3) * KB << 11) + 256u * (n & 7u);
      if constexpr (ES == 2) {
        *reinterpret_cast<uint32_t*>(mr) = bits[1] * 65536u + bits[0];
      } else {
        *reinterpret_cast<uint32_t*>(mr) = bits[0];
        *reinterpret_cast<uint32_t*>(mr + 128) = bits[1];
      }
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t row = (int64_t)n * 16 + in_group + 8 * h;
        if (!FULL && row >= M) continue;
        uint16_t* mr = reinterpret_cast<uint16_t*>(meta_cell0 + row * (K >> 3));
        mr[0] = (uint16_t)bits[h];
        if (ES == 1 && !half_cell) mr[1] = (uint16_t)(bits[h] >> 16);
      }
    }
  }
  count_dropped<COUNT>(lost, dropped);
}

// Units of 16 bytes: a thread has one of the rows r and r + 8, a warp 32 (16, 8) neighbouring ones of 1 (2, 4) rows; neighbouring
// lanes put their metadata together, so that words of the operand order are still written whole.  Half a cell to a thread: for
// matrices of few cells, where compress_kernel's threads go through four vectors one after another on a part of the SMs, and for
// the fused pass at 16-byte boundaries, where the two accesses of a cell meet in its sectors (see compress_any). Bound by the
// latency of that chain, in the fused pass by HBM or the L2.  Us, device, cells and units: compress bf16 360 x 512 1.47, 1.26;
// int8 406 x 128 1.73, 1.37, with the count 2.05, 1.63, fused with prune 1.89, 1.47; 1184 x 1024 1.83, 1.56, 2.10, 1.78, 2.05,
// 1.62.
template <int ES, bool COUNT, bool HW, bool PRUNE>
__global__ void __launch_bounds__(kThreads, kUnitBlocks<COUNT, PRUNE>)
compress_units_kernel(const uint8_t* x, int64_t row_bytes_x, uint8_t* vals, int64_t row_bytes_v, uint8_t* meta, int64_t M, int64_t K,
                      uint32_t row_groups, uint32_t units_pad, int unit_shift, unsigned long long* dropped, int f8, uint8_t* y,
                      int64_t row_bytes_y) {
  wait_for_stream();
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5, odd = lane & 1u;
  const uint32_t rows_of_warp = 32u >> unit_shift, unit = (blockIdx.x << unit_shift) + (lane & ((1u << unit_shift) - 1u));
  const uint32_t thread_row = warp * rows_of_warp + (lane >> unit_shift);  // eight of these to a row group
  const uint32_t in_group = thread_row & 7u, step = gridDim.y * rows_of_warp;
  const bool live_unit = (int64_t)unit * (16 / ES) < K, meta_unit = unit < units_pad;
  // metadata of the unit and its neighbour in the first row of a 128-row block that this thread may write (canonical: in row 0)
  const uint32_t chunk = ES == 2 ? unit >> 1 : unit, KB = ES == 2 ? units_pad >> 4 : units_pad >> 3;
  uint8_t* const meta_unit0 =
      meta + (!HW ? 2 * chunk
                  : (chunk >> 3) * 2048u + 16u * in_group +
                        (ES == 2 ? 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) : 2u * (chunk & 6u) + 128u * odd));
  uint32_t n = blockIdx.y * rows_of_warp + (thread_row >> 3);  // row group, the same for all lanes of a warp
  const int64_t row0 = (int64_t)n * 16 + in_group;
  const uint8_t* xp = x + row0 * row_bytes_x + (int64_t)unit * 16;
  uint8_t* vp = vals + row0 * row_bytes_v + (int64_t)unit * 8;
  uint8_t* yp = PRUNE ? y + row0 * row_bytes_y + (int64_t)unit * 16 : nullptr;
  uint32_t lost = 0;
#pragma unroll 1
  for (; n < row_groups; n += step, xp += (int64_t)step * 16 * row_bytes_x, vp += (int64_t)step * 16 * row_bytes_v) {
    uint4 in[2];
    bool live[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      live[h] = live_unit && (int64_t)n * 16 + in_group + 8 * h < M;
      if (live[h]) in[h] = ld_stream(xp + 8 * h * row_bytes_x);
    }
    uint32_t bits[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      bits[h] = ES == 2 ? 0x44u : 0x4444u;  // padding: positions (0, 1) in all groups
      if (live[h]) {
        uint32_t kept[2], p[4];
        transpose<ES>(in[h], p);
        const Selection<ES> s(p, f8);
        bits[h] = gather_kept<ES>(s, in[h], kept);
        __stcs(reinterpret_cast<uint2*>(vp + 8 * h * row_bytes_v), make_uint2(kept[0], kept[1]));
        if (PRUNE) st_stream(yp + 8 * h * row_bytes_y, s.pruned(p));
        if (COUNT) lost += s.lost();
      }
    }
    if (PRUNE) yp += (int64_t)step * 16 * row_bytes_y;
    uint8_t* const mr = meta_unit0 + ((uint64_t)(n >> 3) * KB << 11) + 256u * (n & 7u);  // (operand order)
    if constexpr (ES == 2) {  // a byte of either row: 16 bits with the neighbour's
      const uint32_t own = bits[1] * 65536u + bits[0], other = __shfl_xor_sync(0xFFFFFFFFu, own, 1);
      const uint32_t word = odd ? own * 256u + other : other * 256u + own;
      if constexpr (HW) {
        if (meta_unit && !odd) *reinterpret_cast<uint32_t*>(mr) = word;
      } else {  // (a row has an even number of units)
        const int64_t row = (int64_t)n * 16 + in_group + 8 * odd;
        if (meta_unit && row < M) *reinterpret_cast<uint16_t*>(meta_unit0 + row * (K >> 3)) = (uint16_t)(odd ? word >> 16 : word);
      }
    } else if constexpr (HW) {  // 16 bits of either row: the even lane writes a word of row r, the odd one of r + 8
      const uint32_t other = __shfl_xor_sync(0xFFFFFFFFu, odd ? bits[0] : bits[1], 1);
      if (meta_unit) *reinterpret_cast<uint32_t*>(mr) = odd ? bits[1] * 65536u + other : other * 65536u + bits[0];
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int64_t row = (int64_t)n * 16 + in_group + 8 * h;
        if (meta_unit && row < M) *reinterpret_cast<uint16_t*>(meta_unit0 + row * (K >> 3)) = (uint16_t)bits[h];
      }
    }
  }
  count_dropped<COUNT>(lost, dropped);
}

// Any alignment: one thread per 8 columns (two groups = one metadata byte), element-wise.
template <typename T>
__global__ void compress_scalar_kernel(const T* __restrict__ x, int64_t ldx, T* __restrict__ vals, int64_t ldv,
                                       uint8_t* __restrict__ meta, int layout, int64_t M, int64_t K,
                                       int64_t rows_pad, int64_t bytes_pad, unsigned long long* dropped, int f8) {
  constexpr int ES = sizeof(T);
  const int64_t total = rows_pad * bytes_pad, KB = bytes_pad >> 4;
  int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= total) return;
  int64_t row = id / bytes_pad, bi = id - row * bytes_pad;  // bi: metadata byte index in the row
  uint32_t mbyte = 0x44u, lost = 0;
  if (row < M && bi < (K >> 3)) {
    mbyte = 0;
    for (int h = 0; h < 2; ++h) {
      const T* src = x + row * ldx + 8 * bi + 4 * h;
      T e[4];
      uint32_t key[4];
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        e[p] = src[p];
        key[p] = ES == 2 ? (uint32_t)((uint16_t)e[p] & 0x7FFFu) : key8((uint32_t)(uint8_t)e[p], f8);
      }
      uint32_t m = keep_mask4(key[0], key[1], key[2], key[3]);
      uint32_t nib = mask_to_nibble(m);
      T* dst = vals + row * ldv + 4 * bi + 2 * h;
      dst[0] = e[nib & 3];
      dst[1] = e[nib >> 2];
      mbyte |= nib << (4 * h);
#pragma unroll
      for (int p = 0; p < 4; ++p) lost += (key[p] != 0 && !((m >> p) & 1u));
    }
  }
  int64_t off = meta_offset<ES>(layout, row, bi >> 1, K, KB) + (bi & 1);
  meta[off] = (uint8_t)mbyte;
  if (dropped != nullptr && lost) atomicAdd(dropped, (unsigned long long)lost);
}

// ---- decompress ---------------------------------------------------------------------------
template <int ES>
__global__ void __launch_bounds__(kThreads) decompress_vec_kernel(const uint8_t* __restrict__ vals, int64_t row_bytes_v,
                                                                  const uint8_t* __restrict__ meta, int layout,
                                                                  uint8_t* __restrict__ y, int64_t row_bytes_y,
                                                                  int64_t M, int64_t K, int64_t chunks_pad) {
  // threads along a row (one 16-column chunk each), blockIdx.y strides over the rows: no division
  const int64_t chunks = K >> 4, KB = chunks_pad >> 3;
  const int64_t chunk = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (chunk >= chunks) return;
  for (int64_t row = blockIdx.y; row < M; row += gridDim.y) {
  uint32_t mbits = *reinterpret_cast<const uint16_t*>(meta + meta_offset<ES>(layout, row, chunk, K, KB));
  if (ES == 2) {
    uint4 v = ld_stream(vals + row * row_bytes_v + chunk * 16);
    uint32_t in[4] = {v.x, v.y, v.z, v.w};
    uint32_t w[8];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      uint32_t nib = (mbits >> (4 * g)) & 0xFu;
      uint64_t both = ((uint64_t)(in[g] & 0xFFFFu) << (16 * (nib & 3))) | ((uint64_t)(in[g] >> 16) << (16 * (nib >> 2)));
      w[2 * g] = (uint32_t)both;
      w[2 * g + 1] = (uint32_t)(both >> 32);
    }
    uint8_t* dst = y + row * row_bytes_y + chunk * 32;
    st_stream(dst, make_uint4(w[0], w[1], w[2], w[3]));
    st_stream(dst + 16, make_uint4(w[4], w[5], w[6], w[7]));
  } else {
    uint2 v = __ldcs(reinterpret_cast<const uint2*>(vals + row * row_bytes_v + chunk * 8));
    uint32_t in[2] = {v.x, v.y};
    uint32_t w[4];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      uint32_t nib = (mbits >> (4 * g)) & 0xFu;
      uint32_t pair = (in[g >> 1] >> (16 * (g & 1))) & 0xFFFFu;
      w[g] = ((pair & 0xFFu) << (8 * (nib & 3))) | ((pair >> 8) << (8 * (nib >> 2)));
    }
    st_stream(y + row * row_bytes_y + chunk * 16, make_uint4(w[0], w[1], w[2], w[3]));
  }
  }
}

template <typename T>
__global__ void decompress_scalar_kernel(const T* __restrict__ vals, int64_t ldv, const uint8_t* __restrict__ meta,
                                         int layout, T* __restrict__ y, int64_t ldy, int64_t M, int64_t K,
                                         int64_t bytes_pad) {
  constexpr int ES = sizeof(T);
  const int64_t KB = bytes_pad >> 4, bytes = K >> 3;
  int64_t id = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (id >= M * bytes) return;
  int64_t row = id / bytes, bi = id - row * bytes;
  uint32_t mbyte = meta[meta_offset<ES>(layout, row, bi >> 1, K, KB) + (bi & 1)];
  for (int h = 0; h < 2; ++h) {
    uint32_t nib = (mbyte >> (4 * h)) & 0xFu;
    const T* src = vals + row * ldv + 4 * bi + 2 * h;
    T* dst = y + row * ldy + 8 * bi + 4 * h;
    T e0 = src[0], e1 = src[1];
#pragma unroll
    for (int p = 0; p < 4; ++p) dst[p] = p == (int)(nib & 3) ? e0 : (p == (int)(nib >> 2) ? e1 : (T)0);
  }
}

// ---- im2col (3x3, stride 1, pad 1, NHWC) ------------------------------------------------------
// Out row = output pixel, out column = (r, s, c).  A block handles the pixels of one image row (n, h):
// blockIdx.x = h, blockIdx.y strides over n, threadIdx = (16-byte vector of channels, filter tap, pixel
// column), so no thread divides anything and a warp writes 512 contiguous bytes.
__global__ void __launch_bounds__(kThreads + 64) im2col_3x3_kernel(const uint8_t* __restrict__ in, uint8_t* __restrict__ out,
                                                                   int64_t row_bytes_out, int64_t Nb, int H, int W,
                                                                   int c_vecs) {
  const int h = blockIdx.x, rs = threadIdx.y, r = rs / 3, s = rs - 3 * r;
  const int hh = h + r - 1;
  const bool row_ok = hh >= 0 && hh < H;
  for (int64_t n = blockIdx.y; n < Nb; n += gridDim.y) {
    const uint8_t* in_row = in + ((n * H + hh) * W) * (int64_t)c_vecs * 16;
    uint8_t* out_row = out + ((n * H + h) * W) * row_bytes_out + (int64_t)rs * c_vecs * 16;
#pragma unroll 4
    for (int w = threadIdx.z; w < W; w += blockDim.z) {
      const int ww = w + s - 1;
      const bool ok = row_ok && ww >= 0 && ww < W;
      for (int cv = threadIdx.x; cv < c_vecs; cv += blockDim.x) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (ok) v = __ldg(reinterpret_cast<const uint4*>(in_row + ((int64_t)ww * c_vecs + cv) * 16));
        st_stream(out_row + w * row_bytes_out + cv * 16, v);
      }
    }
  }
}

// ---- the 1:2 pattern of the TF32 mode (Section 3.2): fp32 storage, one kept value per aligned pair ----
// Metadata: one nibble per pair, 0x4 = first kept, 0xE = second kept (the pair seen as four 16-bit
// halves of which (0,1) or (2,3) survive); canonical K/4 bytes per row, or the operand order of the
// 16-bit types with a nibble standing for a pair (a 2048-byte block = 128 rows x 64 columns).
__device__ __forceinline__ bool keep_second(uint32_t a, uint32_t b) { return (b & 0x7FFFFFFFu) > (a & 0x7FFFFFFFu); }

__global__ void __launch_bounds__(kThreads) prune_f32_kernel(const uint8_t* __restrict__ x, int64_t row_bytes_x, uint8_t* y,
                                                             int64_t row_bytes_y, int64_t vpr, int64_t rows) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= vpr) return;
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < rows; row += (int64_t)gridDim.y * blockDim.y) {
    uint4 v = ld_stream(x + row * row_bytes_x + c * 16);
    const bool s0 = keep_second(v.x, v.y), s1 = keep_second(v.z, v.w);
    st_stream(y + row * row_bytes_y + c * 16, make_uint4(s0 ? 0u : v.x, s0 ? v.y : 0u, s1 ? 0u : v.z, s1 ? v.w : 0u));
  }
}

// Work unit: 8 columns (four pairs) = 32 bytes in, 16 bytes of values and 16 bits of metadata out.
template <bool HW>
__global__ void __launch_bounds__(kThreads) compress_f32_kernel(const uint8_t* __restrict__ x, int64_t row_bytes_x,
                                                                uint8_t* __restrict__ vals, int64_t row_bytes_v,
                                                                uint8_t* __restrict__ meta, int64_t M, int64_t K,
                                                                int64_t rows_pad, int64_t chunks_pad,
                                                                unsigned long long* dropped) {
  const uint32_t chunk = blockIdx.x * blockDim.x + threadIdx.x, chunks = (uint32_t)(K >> 3), KB = (uint32_t)(chunks_pad >> 3);
  const int64_t moff = HW ? (int64_t)(chunk >> 3) * 2048 + 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) : (int64_t)chunk * 2;
  uint32_t lost = 0;
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < rows_pad;
       row += (int64_t)gridDim.y * blockDim.y) {
    if (chunk >= (uint32_t)chunks_pad) continue;
    uint32_t mbits = 0x4444u;
    if (row < M && chunk < chunks) {
      const uint8_t* src = x + row * row_bytes_x + (int64_t)chunk * 32;
      const uint4 a = ld_stream(src), b = ld_stream(src + 16);
      const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
      uint32_t out[4];
      mbits = 0;
#pragma unroll
      for (int g = 0; g < 4; ++g) {
        const bool sec = keep_second(w[2 * g], w[2 * g + 1]);
        out[g] = sec ? w[2 * g + 1] : w[2 * g];
        mbits |= (sec ? 0xEu : 0x4u) << (4 * g);
        lost += ((sec ? w[2 * g] : w[2 * g + 1]) & 0x7FFFFFFFu) != 0;
      }
      st_stream(vals + row * row_bytes_v + (int64_t)chunk * 16, make_uint4(out[0], out[1], out[2], out[3]));
    }
    const uint32_t r = (uint32_t)row & 127u;
    uint8_t* mr = HW ? meta + (row >> 7) * ((int64_t)KB * 2048) + (16u * (r & 7u) + 2u * ((r >> 3) & 1u) + 256u * (r >> 4))
                     : meta + row * (K >> 2);
    *reinterpret_cast<uint16_t*>(mr + moff) = (uint16_t)mbits;
  }
  if (dropped != nullptr && lost) atomicAdd(dropped, (unsigned long long)lost);
}

template <bool HW>
__global__ void __launch_bounds__(kThreads) decompress_f32_kernel(const uint8_t* __restrict__ vals, int64_t row_bytes_v,
                                                                  const uint8_t* __restrict__ meta, uint8_t* __restrict__ y,
                                                                  int64_t row_bytes_y, int64_t M, int64_t K,
                                                                  int64_t chunks_pad) {
  const uint32_t chunk = blockIdx.x * blockDim.x + threadIdx.x, chunks = (uint32_t)(K >> 3), KB = (uint32_t)(chunks_pad >> 3);
  if (chunk >= chunks) return;
  const int64_t moff = HW ? (int64_t)(chunk >> 3) * 2048 + 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) : (int64_t)chunk * 2;
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < M; row += (int64_t)gridDim.y * blockDim.y) {
    const uint32_t r = (uint32_t)row & 127u;
    const uint8_t* mr = HW ? meta + (row >> 7) * ((int64_t)KB * 2048) + (16u * (r & 7u) + 2u * ((r >> 3) & 1u) + 256u * (r >> 4))
                           : meta + row * (K >> 2);
    const uint32_t mbits = *reinterpret_cast<const uint16_t*>(mr + moff);
    const uint4 v = ld_stream(vals + row * row_bytes_v + (int64_t)chunk * 16);
    const uint32_t in[4] = {v.x, v.y, v.z, v.w};
    uint32_t w[8];
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      const bool sec = (((mbits >> (4 * g)) & 3u) >> 1) != 0;
      w[2 * g] = sec ? 0u : in[g];
      w[2 * g + 1] = sec ? in[g] : 0u;
    }
    uint8_t* dst = y + row * row_bytes_y + (int64_t)chunk * 32;
    st_stream(dst, make_uint4(w[0], w[1], w[2], w[3]));
    st_stream(dst + 16, make_uint4(w[4], w[5], w[6], w[7]));
  }
}

inline unsigned blocks_for(int64_t total, int per_block) { return (unsigned)((total + per_block - 1) / per_block); }

}  // namespace

static sp24_status validate_matrix_args(sp24_dtype t, int64_t M, int64_t K, int64_t k_multiple) {
  SP24_RETURN_IF(!is_ab_type(t), SP24_ERR_DTYPE);
  SP24_RETURN_IF(M < 0 || K < 0 || K % k_multiple != 0, SP24_ERR_SHAPE);
  return SP24_OK;
}

}  // namespace sp24

using namespace sp24;

// FP32 storage = the 1:2 pattern of the TF32 mode; vectorised paths only (16-byte aligned, K % 8 == 0).
static sp24_status validate_f32(int64_t M, int64_t K) {
  SP24_RETURN_IF(M < 0 || K < 0 || K % 8 != 0, SP24_ERR_SHAPE);
  return SP24_OK;
}

static dim3 f32_grid(int64_t units, int64_t rows, dim3& block) {
  block = dim3(256, 1, 1);
  if (units <= 128) block = dim3(units <= 32 ? 32 : (units <= 64 ? 64 : 128), 1, 1);
  block.y = kThreads / block.x;
  int64_t gy = (rows + block.y - 1) / block.y;
  if (gy > 32768) gy = 32768;
  return dim3((unsigned)((units + block.x - 1) / block.x), (unsigned)gy, 1);
}

extern "C" sp24_status sp24_prune(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx, void* y,
                                  int64_t ldy, void* stream) {
  if (t == SP24_F32) {
    sp24_status sf = validate_f32(M, K);
    if (sf != SP24_OK) return sf;
    if (M == 0 || K == 0) return SP24_OK;
    SP24_RETURN_IF(x == nullptr || y == nullptr, SP24_ERR_NULL);
    SP24_RETURN_IF(ldx < K || ldy < K || ldx % 4 || ldy % 4, SP24_ERR_STRIDE);
    SP24_RETURN_IF(!aligned16(x) || !aligned16(y), SP24_ERR_ALIGN);
    if ((sf = check_arch()) != SP24_OK) return sf;
    dim3 block, grid = f32_grid(K / 4, M, block);
    prune_f32_kernel<<<grid, block, 0, static_cast<cudaStream_t>(stream)>>>((const uint8_t*)x, ldx * 4, (uint8_t*)y, ldy * 4,
                                                                             K / 4, M);
    return cuda_status(cudaGetLastError());
  }
  sp24_status st = validate_matrix_args(t, M, K, 4);
  if (st != SP24_OK) return st;
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(x == nullptr || y == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldx < K || ldy < K, SP24_ERR_STRIDE);
  if ((st = check_arch()) != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int es = elem_bytes(t), f8 = is_fp8(t) ? 1 : 0;
  const bool vec = aligned16(x) && aligned16(y) && (ldx * es) % 16 == 0 && (ldy * es) % 16 == 0 && (K * es) % 16 == 0 &&
                   row_offsets_fit(K, es, SP24_META_CANONICAL);
  if (vec) {
    constexpr int UNROLL = 4;
    int64_t vpr = K * es / 16, rows = M;
    if (ldx == K && ldy == K && vpr < 256 * UNROLL) {  // packed and short rows: fold rows into long ones
      int64_t fold = 1;
      while (vpr * fold * 2 <= 256 * UNROLL && rows % 2 == 0) { fold *= 2; rows /= 2; }
      vpr *= fold;
    }
    RowLaunch L(vpr, rows, UNROLL);
    int64_t rbx = ldx == K && ldy == K ? vpr * 16 : ldx * es, rby = ldx == K && ldy == K ? vpr * 16 : ldy * es;
    if (es == 2)
      return launch_streaming(Kernel<prune_vec_kernel<2, UNROLL>>{}, L.grid, L.block, s, (const uint8_t*)x, rbx, (uint8_t*)y, rby,
                               vpr, rows, f8);
    else
      return launch_streaming(Kernel<prune_vec_kernel<1, UNROLL>>{}, L.grid, L.block, s, (const uint8_t*)x, rbx, (uint8_t*)y, rby,
                               vpr, rows, f8);
  } else {
    int64_t gpr = K / 4, total = M * gpr;
    unsigned blocks = blocks_for(total, kThreads);
    if (es == 2)
      prune_scalar_kernel<uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, (uint16_t*)y, ldy, gpr, total, 0);
    else
      prune_scalar_kernel<int8_t><<<blocks, kThreads, 0, s>>>((const int8_t*)x, ldx, (int8_t*)y, ldy, gpr, total, f8);
  }
  return cuda_status(cudaGetLastError());
}

namespace sp24 {
namespace {

// compress (y == nullptr) or fused prune + compress (y = pruned matrix, vector kernels only: returns
// SP24_ERR_UNSUPPORTED when they cannot take the operands) for the 2:4 types.
sp24_status compress_any(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx, void* y, int64_t ldy,
                         void* vals, int64_t ldv, void* meta, sp24_meta_layout l, unsigned long long* dropped,
                         void* stream) {
  sp24_status st = validate_matrix_args(t, M, K, 8);
  if (st != SP24_OK) return st;
  SP24_RETURN_IF(l != SP24_META_CANONICAL && l != SP24_META_TCGEN05, SP24_ERR_UNSUPPORTED);
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(x == nullptr || vals == nullptr || meta == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldx < K || ldv < K / 2, SP24_ERR_STRIDE);
  if ((st = check_arch()) != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int es = elem_bytes(t), f8 = is_fp8(t) ? 1 : 0;
  const bool hw = l == SP24_META_TCGEN05;
  const int64_t rows_pad = hw ? (M + 127) / 128 * 128 : M;
  const int64_t k_pad = hw ? (K + 255) / 256 * 256 : K;
  const bool vec = K % 16 == 0 && aligned16(x) && aligned16(vals) && aligned16(meta) && (ldx * es) % 16 == 0 &&
                   (ldv * es) % (8 * es) == 0 && row_offsets_fit(K, es, l);
  if (vec) {
    const uint8_t* xs = (const uint8_t*)x;
    uint8_t *vs = (uint8_t*)vals, *ms = (uint8_t*)meta, *ys = (uint8_t*)y;
    // Blocks along the rows, for warps with 2^shift units of a row.  A matrix of moderate size is bound by instructions: about two
    // rounds of the blocks that fit the SMs take all rows (whole rows of blocks, so a few blocks may make a third), and the set-up
    // of a block is paid for once.  A large one is bound by HBM and wants the loads of all its blocks in flight.  The line, 160 MB
    // of traffic, is that of apply_mask + compress and of the fused pass.  Us, device, a block for every row step and two rounds,
    // at MB of traffic: apply_mask + compress bf16 4096 x 4096 (50) 13.4, 13.2; 12288 x 3072 (112) 35.8, 35.0; 12288 x 4096 (150)
    // 49.8, 49.6; 8192 x 8192 (200) 68.4, 69.2; 16384 x 8192 (400) 141, 149; int8 8192 x 8192 (104) 38.7, 37.5; fused bf16 4096 x
    // 4096 (82) 10.0, 9.4; 12288 x 3072 (184) 29.8, 31.5; int8 12288 x 4096 (126) 21.7, 19.9; 8192 x 8192 (168) 28.9, 29.9; alone
    // on operands that stay in the L2 bf16 12288 x 3072 (112) 14.8, 15.8, int8 9000 x 16384 (229) 49.2, 42.6.
    const int64_t groups = (rows_pad + 15) / 16, moved = M * K * es * (y ? 5 : 3) / 2 + M * K / 8;
    auto row_steps = [&](int shift, int64_t columns, int blocks_of_sm) {
      int64_t steps = (groups + (32 >> shift) - 1) / (32 >> shift);
      if (steps > 32768) steps = 32768;
      const int64_t two_rounds = (2 * blocks_of_sm * sm_count() + columns - 1) / columns;
      return moved <= (int64_t)160 << 20 && steps > two_rounds ? two_rounds : steps;
    };
    const int64_t cols = es == 2 ? 16 : 32, cells_pad = (k_pad + cols - 1) / cols;
    const bool whole_cells = K % cols == 0;
    auto by32 = [&](const void* p, int64_t ld) { return whole_cells && reinterpret_cast<uintptr_t>(p) % 32 == 0 && ld * es % 32 == 0; };
    const int shift = (cells_pad - 1) % 16 < 8 ? 3 : 4;  // cells of a row to a warp: 8 or 16, whichever leaves fewer lanes idle
    const int64_t units = (cells_pad + (1 << shift) - 1) >> shift;
    const bool full = rows_pad == M && M % 16 == 0 && k_pad == K && whole_cells && cells_pad == units << shift;
    const int64_t steps = row_steps(shift, units, es == 2 && !dropped && !y ? kCompressBlocks<2, false, false> : kCompressBlocks<1, true, true>);
    // Fewer blocks of cells than three for two SMs (3.6 MB where no lanes are idle): units of half a cell.  Cells over units, means of
    // 3 to 12 matrices, bf16 and int8: compression alone 0.3 to 0.8 MB 1.16, 1.22; 1.2 to 1.8 MB 0.97, 0.99; 2.4 to 3.6 MB 1.02,
    // 1.06; 3.6 to 4.9 MB 0.98, 1.01; 6.5 to 10 MB 0.90, 0.91; fused and a product behind it 1.2 to 1.8 MB 1.01, 1.01; 2.4 to 3.6 MB
    // 1.05, 1.02; 3.6 to 4.9 MB 0.98, 1.01; 6.5 to 10 MB 0.98, 0.98.
    // The fused pass on rows that are not at 32-byte boundaries too, up to 40 M elements, 64 M where they end in half a cell:
    // each of a cell's two stores would leave halves of sectors to the other.  (Whole 8-bit matrices are faster in cells all the
    // same.)  Us, 16-byte vectors of one row, cells and units: bf16 3072 x 1024 3.28, 3.51, 2.98; 4096 x 4096 11.6, 13.0, 10.1;
    // 12928 x 1488 14.5, 15.9, 12.9; 12288 x 3072 30.7, 31.3, 31.1; 67606 x 7296 449, 408, 420; int8 4100 x 4112 9.9, 8.3, 7.9;
    // 4096 x 4096 7.3, 6.6, 7.1; 7468 x 9312 in place 34.6, 33.4, 35.9; with half a cell 32243 x 1040 21.8, 18.0, 16.5; 9098 x
    // 4752 22.1, 25.9, 20.3; 17858 x 8336 75.4, 73.7, 74.6.
    const bool split_stores = y && !(by32(x, ldx) && by32(y, ldy)) && (es == 2 || !full);
    if (2 * units * steps < 3 * sm_count() || (split_stores && M * K <= (int64_t)(whole_cells ? 40 : 64) << 20)) {
      const int64_t units_pad = k_pad / (16 / es);
      auto padded = [&](int log) { return (units_pad + (1 << log) - 1) >> log << log; };
      const int64_t most = padded(3) + units_pad / 16;  // 32, 16 or 8 units of a row to a warp: the most of which few lanes are idle
      const int log = padded(5) <= most ? 5 : padded(4) <= most ? 4 : 3;
      const int64_t columns = padded(log) >> log;
      const dim3 grid((unsigned)columns, (unsigned)row_steps(log, columns, dropped && y ? kUnitBlocks<true, true> : kUnitBlocks<false, false>), 1);
      auto launch = [&](auto kernel) {
        return launch_streaming(kernel, grid, dim3(kThreads), s, xs, ldx * es, vs, ldv * es, ms, M, K, (uint32_t)groups, (uint32_t)units_pad, log,
                                dropped, f8, ys, ldy * es);
      };
#define SP24_CU(V, COUNT, HW, PRUNE) \
  case V:                            \
    return es == 2 ? launch(Kernel<compress_units_kernel<2, COUNT, HW, PRUNE>>{}) : launch(Kernel<compress_units_kernel<1, COUNT, HW, PRUNE>>{});
      switch ((y ? 4 : 0) | (dropped ? 2 : 0) | (hw ? 1 : 0)) {
        SP24_CU(0, false, false, false)
        SP24_CU(1, false, true, false)
        SP24_CU(2, true, false, false)
        SP24_CU(3, true, true, false)
        SP24_CU(4, false, false, true)
        SP24_CU(5, false, true, true)
        SP24_CU(6, true, false, true)
        default:
          SP24_CU(7, true, true, true)
      }
#undef SP24_CU
    }
    const dim3 grid((unsigned)units, (unsigned)steps, 1);
    const int wide = (by32(x, ldx) ? kWideX : 0) | (y && by32(y, ldy) ? kWideY : 0) | (whole_cells && ldv * es % 16 == 0 ? kWideVals : 0);
    const int variant = (y ? 8 : 0) | (dropped ? 4 : 0) | (hw ? 2 : 0) | (full ? 1 : 0);
    auto launch = [&](auto kernel) {
      return launch_streaming(kernel, grid, dim3(kThreads), s, xs, ldx * es, vs, ldv * es, ms, M, K, (uint32_t)groups, (uint32_t)cells_pad, shift,
                              wide, dropped, f8, ys, ldy * es);
    };
#define SP24_CV(V, COUNT, HW, FULL, PRUNE) \
  case V:                                  \
    return es == 2 ? launch(Kernel<compress_kernel<2, COUNT, HW, FULL, PRUNE>>{}) : launch(Kernel<compress_kernel<1, COUNT, HW, FULL, PRUNE>>{});
    switch (variant) {
      SP24_CV(0, false, false, false, false)
      SP24_CV(1, false, false, true, false)
      SP24_CV(2, false, true, false, false)
      SP24_CV(3, false, true, true, false)
      SP24_CV(4, true, false, false, false)
      SP24_CV(5, true, false, true, false)
      SP24_CV(6, true, true, false, false)
      SP24_CV(7, true, true, true, false)
      SP24_CV(8, false, false, false, true)
      SP24_CV(9, false, false, true, true)
      SP24_CV(10, false, true, false, true)
      SP24_CV(11, false, true, true, true)
      SP24_CV(12, true, false, false, true)
      SP24_CV(13, true, false, true, true)
      SP24_CV(14, true, true, false, true)
      default:
        SP24_CV(15, true, true, true, true)
    }
#undef SP24_CV
  } else {
    if (y != nullptr) return SP24_ERR_UNSUPPORTED;
    int64_t bytes_pad = k_pad / 8, total = rows_pad * bytes_pad;
    unsigned blocks = blocks_for(total, kThreads);
    if (es == 2)
      compress_scalar_kernel<uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, (uint16_t*)vals, ldv,
                                                                   (uint8_t*)meta, (int)l, M, K, rows_pad, bytes_pad,
                                                                   dropped, 0);
    else
      compress_scalar_kernel<int8_t><<<blocks, kThreads, 0, s>>>((const int8_t*)x, ldx, (int8_t*)vals, ldv,
                                                                 (uint8_t*)meta, (int)l, M, K, rows_pad, bytes_pad,
                                                                 dropped, f8);
  }
  return cuda_status(cudaGetLastError());
}

}  // namespace
}  // namespace sp24

extern "C" sp24_status sp24_compress(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx, void* vals,
                                     int64_t ldv, void* meta, sp24_meta_layout l, unsigned long long* dropped,
                                     void* stream) {
  if (t == SP24_F32) {
    sp24_status sf = validate_f32(M, K);
    if (sf != SP24_OK) return sf;
    SP24_RETURN_IF(l != SP24_META_CANONICAL && l != SP24_META_TCGEN05, SP24_ERR_UNSUPPORTED);
    if (M == 0 || K == 0) return SP24_OK;
    SP24_RETURN_IF(x == nullptr || vals == nullptr || meta == nullptr, SP24_ERR_NULL);
    SP24_RETURN_IF(ldx < K || ldv < K / 2 || ldx % 4 || ldv % 4, SP24_ERR_STRIDE);
    SP24_RETURN_IF(!aligned16(x) || !aligned16(vals) || !aligned16(meta), SP24_ERR_ALIGN);
    if ((sf = check_arch()) != SP24_OK) return sf;
    const bool hw = l == SP24_META_TCGEN05;
    const int64_t rows_pad = hw ? (M + 127) / 128 * 128 : M, k_pad = hw ? (K + 127) / 128 * 128 : K;
    dim3 block, grid = f32_grid(k_pad / 8, rows_pad, block);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (hw)
      compress_f32_kernel<true><<<grid, block, 0, s>>>((const uint8_t*)x, ldx * 4, (uint8_t*)vals, ldv * 4, (uint8_t*)meta,
                                                       M, K, rows_pad, k_pad / 8, dropped);
    else
      compress_f32_kernel<false><<<grid, block, 0, s>>>((const uint8_t*)x, ldx * 4, (uint8_t*)vals, ldv * 4, (uint8_t*)meta,
                                                        M, K, rows_pad, k_pad / 8, dropped);
    return cuda_status(cudaGetLastError());
  }
  return compress_any(t, M, K, x, ldx, nullptr, 0, vals, ldv, meta, l, dropped, stream);
}

extern "C" sp24_status sp24_prune_compress(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx, void* y,
                                           int64_t ldy, void* vals, int64_t ldv, void* meta, sp24_meta_layout l,
                                           unsigned long long* dropped, void* stream) {
  const int es = elem_bytes(t);
  const bool fused = is_ab_type(t) && y != nullptr && aligned16(y) && es > 0 && (ldy * es) % 16 == 0 && ldy >= K;
  if (fused) {
    const sp24_status st = compress_any(t, M, K, x, ldx, y, ldy, vals, ldv, meta, l, dropped, stream);
    if (st != SP24_ERR_UNSUPPORTED) return st;
  }
  // no fused kernel for this case (1:2 pattern, or operands the vector kernels cannot take): two passes.
  // compress reads x before prune may overwrite it (y may be x).
  sp24_status st = sp24_compress(t, M, K, x, ldx, vals, ldv, meta, l, dropped, stream);
  if (st != SP24_OK) return st;
  return sp24_prune(t, M, K, x, ldx, y, ldy, stream);
}

extern "C" sp24_status sp24_decompress(sp24_dtype t, int64_t M, int64_t K, const void* vals, int64_t ldv,
                                       const void* meta, sp24_meta_layout l, void* y, int64_t ldy, void* stream) {
  if (t == SP24_F32) {
    sp24_status sf = validate_f32(M, K);
    if (sf != SP24_OK) return sf;
    SP24_RETURN_IF(l != SP24_META_CANONICAL && l != SP24_META_TCGEN05, SP24_ERR_UNSUPPORTED);
    if (M == 0 || K == 0) return SP24_OK;
    SP24_RETURN_IF(y == nullptr || vals == nullptr || meta == nullptr, SP24_ERR_NULL);
    SP24_RETURN_IF(ldy < K || ldv < K / 2 || ldy % 4 || ldv % 4, SP24_ERR_STRIDE);
    SP24_RETURN_IF(!aligned16(y) || !aligned16(vals) || !aligned16(meta), SP24_ERR_ALIGN);
    if ((sf = check_arch()) != SP24_OK) return sf;
    const bool hw = l == SP24_META_TCGEN05;
    const int64_t k_pad = hw ? (K + 127) / 128 * 128 : K;
    dim3 block, grid = f32_grid(K / 8, M, block);
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    if (hw)
      decompress_f32_kernel<true><<<grid, block, 0, s>>>((const uint8_t*)vals, ldv * 4, (const uint8_t*)meta, (uint8_t*)y,
                                                         ldy * 4, M, K, k_pad / 8);
    else
      decompress_f32_kernel<false><<<grid, block, 0, s>>>((const uint8_t*)vals, ldv * 4, (const uint8_t*)meta, (uint8_t*)y,
                                                          ldy * 4, M, K, k_pad / 8);
    return cuda_status(cudaGetLastError());
  }
  sp24_status st = validate_matrix_args(t, M, K, 8);
  if (st != SP24_OK) return st;
  SP24_RETURN_IF(l != SP24_META_CANONICAL && l != SP24_META_TCGEN05, SP24_ERR_UNSUPPORTED);
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(y == nullptr || vals == nullptr || meta == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldy < K || ldv < K / 2, SP24_ERR_STRIDE);
  if ((st = check_arch()) != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int es = elem_bytes(t);
  const bool hw = l == SP24_META_TCGEN05;
  const int64_t k_pad = hw ? (K + 255) / 256 * 256 : K;
  const bool vec = K % 16 == 0 && aligned16(y) && aligned16(vals) && aligned16(meta) && (ldy * es) % 16 == 0 &&
                   (ldv * es) % (8 * es) == 0;
  if (vec) {
    const dim3 blocks((unsigned)((K / 16 + kThreads - 1) / kThreads), (unsigned)(M < 16384 ? M : 16384), 1);
    if (es == 2)
      decompress_vec_kernel<2><<<blocks, kThreads, 0, s>>>((const uint8_t*)vals, ldv * es, (const uint8_t*)meta, (int)l,
                                                           (uint8_t*)y, ldy * es, M, K, k_pad / 16);
    else
      decompress_vec_kernel<1><<<blocks, kThreads, 0, s>>>((const uint8_t*)vals, ldv * es, (const uint8_t*)meta, (int)l,
                                                           (uint8_t*)y, ldy * es, M, K, k_pad / 16);
  } else {
    int64_t total = M * (K / 8);
    unsigned blocks = blocks_for(total, kThreads);
    if (es == 2)
      decompress_scalar_kernel<uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)vals, ldv, (const uint8_t*)meta,
                                                                     (int)l, (uint16_t*)y, ldy, M, K, k_pad / 8);
    else
      decompress_scalar_kernel<int8_t><<<blocks, kThreads, 0, s>>>((const int8_t*)vals, ldv, (const uint8_t*)meta,
                                                                   (int)l, (int8_t*)y, ldy, M, K, k_pad / 8);
  }
  return cuda_status(cudaGetLastError());
}

extern "C" sp24_status sp24_im2col_nhwc_3x3(sp24_dtype t, int64_t Nb, int64_t H, int64_t W, int64_t C, const void* in,
                                            void* out, int64_t ldo, void* stream) {
  SP24_RETURN_IF(!is_ab_type(t), SP24_ERR_DTYPE);
  SP24_RETURN_IF(Nb < 0 || H < 0 || W < 0 || C < 0 || H > (1 << 30) || W > (1 << 30), SP24_ERR_SHAPE);
  const int es = elem_bytes(t);
  SP24_RETURN_IF((C * es) % 16 != 0, SP24_ERR_SHAPE);
  if (Nb == 0 || H == 0 || W == 0 || C == 0) return SP24_OK;
  SP24_RETURN_IF(in == nullptr || out == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldo < 9 * C || (ldo * es) % 16 != 0, SP24_ERR_STRIDE);
  SP24_RETURN_IF(!aligned16(in) || !aligned16(out), SP24_ERR_ALIGN);
  sp24_status st = check_arch();
  if (st != SP24_OK) return st;
  const int64_t c_vecs = C * es / 16;
  SP24_RETURN_IF(c_vecs > (1 << 24), SP24_ERR_SHAPE);
  const unsigned bx = (unsigned)(c_vecs < 32 ? c_vecs : 32);
  unsigned bz = 288u / (9u * bx);
  bz = bz < 1 ? 1 : (bz > (unsigned)W ? (unsigned)W : bz);
  const dim3 block(bx, 9, bz), grid((unsigned)H, (unsigned)(Nb < 65535 ? Nb : 65535), 1);
  im2col_3x3_kernel<<<grid, block, 0, static_cast<cudaStream_t>(stream)>>>((const uint8_t*)in, (uint8_t*)out, ldo * es, Nb,
                                                                           (int)H, (int)W, (int)c_vecs);
  return cuda_status(cudaGetLastError());
}
