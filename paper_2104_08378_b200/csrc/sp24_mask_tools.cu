// Tools around the pruning step of the workflow (Section 4.1 and Section 6 of arXiv 2104.08378):
//   sp24_kept_magnitude  total magnitude that 2:4 pruning keeps, optionally under a column
//                        permutation: the figure of merit of the channel permutations of Section 4.1;
//   sp24_apply_mask      re-imposes a fixed 2:4 pattern (given as metadata) on changed weights: what
//                        sparse retraining (step 3) does after every update;
//   sp24_prune_2d        2:4 along rows AND columns of every 4x4 block, so that the transposed matrix
//                        is 2:4 as well (Section 6), by exhaustive search over the 90 such patterns.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include "sp24_common.cuh"

namespace sp24 {
namespace {

__device__ __forceinline__ uint32_t keep_mask4(uint32_t k0, uint32_t k1, uint32_t k2, uint32_t k3) {
  uint32_t c01 = k0 >= k1, c02 = k0 >= k2, c03 = k0 >= k3;
  uint32_t c12 = k1 >= k2, c13 = k1 >= k3, c23 = k2 >= k3;
  uint32_t b0 = 3u - (c01 + c02 + c03), b1 = c01 + 2u - (c12 + c13);
  uint32_t b2 = c02 + c12 + 1u - c23, b3 = c03 + c13 + c23;
  return (b0 < 2u) | ((b1 < 2u) << 1) | ((b2 < 2u) << 2) | ((b3 < 2u) << 3);
}

template <typename T>
__device__ __forceinline__ uint32_t key_of(T e) {
  return sizeof(T) == 2 ? (uint32_t)((uint16_t)e & 0x7FFFu) : (uint32_t)abs((int)(int8_t)e);
}

// |value| as a float, exact for all three storage types.  DT: 0 fp16, 1 bf16, 2 int8.
template <int DT, typename T>
__device__ __forceinline__ float magnitude_of(T e) {
  if (DT == 2) return (float)abs((int)(int8_t)e);
  uint16_t bits = (uint16_t)e & 0x7FFFu;
  if (DT == 0) return __half2float(*reinterpret_cast<__half*>(&bits));
  return __bfloat162float(*reinterpret_cast<__nv_bfloat16*>(&bits));
}

// ---- kept magnitude -------------------------------------------------------------------------------
// One block sums its threads' partial sums and adds them to *result with one atomic.
__device__ __forceinline__ void block_add(double sum, double* result) {
  __shared__ double part[kThreads / 32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xFFFFFFFFu, sum, o);
  const int t = threadIdx.x;
  if ((t & 31) == 0) part[t >> 5] = sum;
  __syncthreads();
  if (t == 0) {
    double s = 0.0;
#pragma unroll
    for (int w = 0; w < kThreads / 32; ++w) s += part[w];
    atomicAdd(result, s);
  }
}

template <int DT, typename T>
__global__ void __launch_bounds__(kThreads) kept_magnitude_kernel(const T* __restrict__ x, int64_t ldx, int64_t M,
                                                                  int64_t groups, const int32_t* __restrict__ perm,
                                                                  double* result) {
  double sum = 0.0;
  const int64_t total = M * groups;
  for (int64_t id = (int64_t)blockIdx.x * kThreads + threadIdx.x; id < total; id += (int64_t)gridDim.x * kThreads) {
    const int64_t row = id / groups, g = id - row * groups;
    T e[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) {
      const int64_t col = perm ? (int64_t)perm[4 * g + p] : 4 * g + p;
      e[p] = x[row * ldx + col];
    }
    const uint32_t m = keep_mask4(key_of(e[0]), key_of(e[1]), key_of(e[2]), key_of(e[3]));
#pragma unroll
    for (int p = 0; p < 4; ++p)
      if ((m >> p) & 1u) sum += (double)magnitude_of<DT>(e[p]);
  }
  block_add(sum, result);
}

// Kept magnitude of the groups held in one 16-byte vector (two groups of a 16-bit type, four of int8).
template <int DT>
__device__ __forceinline__ double kept_in_vector(uint4 v) {
  double sum = 0.0;
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  if (DT == 2) {
#pragma unroll
    for (int g = 0; g < 4; ++g) {
      uint32_t a = __vabs4(w[g]);  // -128 -> 128
      uint32_t k0 = a & 0xFFu, k1 = (a >> 8) & 0xFFu, k2 = (a >> 16) & 0xFFu, k3 = a >> 24;
      uint32_t m = keep_mask4(k0, k1, k2, k3);
      uint32_t kept = ((m & 1u) ? k0 : 0u) + ((m & 2u) ? k1 : 0u) + ((m & 4u) ? k2 : 0u) + ((m & 8u) ? k3 : 0u);
      sum += (double)kept;  // integers: exact
    }
  } else {
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const uint32_t lo = w[2 * g] & 0x7FFF7FFFu, hi = w[2 * g + 1] & 0x7FFF7FFFu;
      const uint32_t k[4] = {lo & 0xFFFFu, lo >> 16, hi & 0xFFFFu, hi >> 16};
      const uint32_t m = keep_mask4(k[0], k[1], k[2], k[3]);
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if ((m >> p) & 1u) sum += (double)magnitude_of<DT>((uint16_t)k[p]);
    }
  }
  return sum;
}

// Identity permutation, 16-byte aligned rows: threads along a row, one vector per thread and row step.
template <int DT>
__global__ void __launch_bounds__(kThreads) kept_magnitude_vec_kernel(const uint8_t* __restrict__ x, int64_t row_bytes,
                                                                      int64_t M, int64_t vpr, double* result) {
  double sum = 0.0;
  const int64_t c = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (c < vpr) {
    for (int64_t row = blockIdx.y; row < M; row += gridDim.y)
      sum += kept_in_vector<DT>(__ldcs(reinterpret_cast<const uint4*>(x + row * row_bytes + c * 16)));
  }
  block_add(sum, result);
}

// Column permutation, 16-byte aligned rows of at most 48 KB: a block copies one row into shared memory
// with coalesced vector loads and gathers the permuted groups from there.
template <int DT, typename T>
__global__ void __launch_bounds__(kThreads) kept_magnitude_perm_kernel(const uint8_t* __restrict__ x, int64_t row_bytes,
                                                                       int64_t M, int64_t K,
                                                                       const int32_t* __restrict__ perm, double* result) {
  extern __shared__ uint4 row_buf[];
  const T* row_elems = reinterpret_cast<const T*>(row_buf);
  const int64_t vpr = K * (int64_t)sizeof(T) / 16, groups = K / 4;
  double sum = 0.0;
  for (int64_t row = blockIdx.x; row < M; row += gridDim.x) {
    for (int64_t c = threadIdx.x; c < vpr; c += kThreads)
      row_buf[c] = __ldcs(reinterpret_cast<const uint4*>(x + row * row_bytes + c * 16));
    __syncthreads();
    for (int64_t g = threadIdx.x; g < groups; g += kThreads) {
      const int4 pc = *reinterpret_cast<const int4*>(perm + 4 * g);
      T e[4] = {row_elems[pc.x], row_elems[pc.y], row_elems[pc.z], row_elems[pc.w]};
      const uint32_t m = keep_mask4(key_of(e[0]), key_of(e[1]), key_of(e[2]), key_of(e[3]));
#pragma unroll
      for (int p = 0; p < 4; ++p)
        if ((m >> p) & 1u) sum += (double)magnitude_of<DT>(e[p]);
    }
    __syncthreads();
  }
  block_add(sum, result);
}

// ---- apply mask -----------------------------------------------------------------------------------
// A metadata nibble indexes a table of byte-permute selectors that copy the two positions it names and zero the others (16 words:
// no two of them share a bank).
template <int ES>
__device__ __forceinline__ void mask_selectors(uint32_t (&table)[16], uint32_t t) {
  if (t < 16) {
    const uint32_t keep = (1u << (t & 3u)) | (1u << (t >> 2));
    // selector nibble 4 = a zero byte of the second operand; 16-bit types: a selector for each of a group's two words
    uint32_t sel = 0;
#pragma unroll
    for (uint32_t i = 0; i < 4; ++i)
      sel |= ES == 2 ? ((keep >> i) & 1u ? (i & 1u ? 0x32u : 0x10u) : 0x44u) << (8 * i) : ((keep >> i) & 1u ? i : 4u) << (4 * i);
    table[t] = sel;
  }
  __syncthreads();
}

// Rows of whole cells (32 bytes) at 32-byte boundaries: cells of two rows to a thread and metadata addresses as in compress_kernel,
// so that a thread's metadata is one or two words.
// Bound by HBM, by the instructions where the rows are short.  The result is stored without an evict-first hint: it is
// compressed next, and as much of it as fits is then read from the L2.  With 16-byte units of one row, a metadata byte or two read
// for each, a vector took 59 instructions (int8 76).  Us, device, with the compression, units and cells: bf16 49152 x 256 18.4,
// 13.4; 16102 x 1088 21.8, 20.4; 4096 x 4096 18.3, 17.8; 12288 x 3072 36.1, 35.8; int8 49152 x 256 17.4,
// 9.1; 12288 x 3072 24.7, 24.1.  (Cells by two 16-byte accesses at other boundaries: 5 to 20 % slower than the units.)
template <int ES, bool HW, bool FULL>
__global__ void __launch_bounds__(kThreads, 5) apply_mask_vec_kernel(const uint8_t* w, int64_t row_bytes_w, const uint8_t* meta,
                                                                     uint8_t* y, int64_t row_bytes_y, int64_t M, int64_t K,
                                                                     uint32_t row_groups, uint32_t KB, int cell_shift) {
  constexpr uint32_t kCols = ES == 2 ? 16 : 32;  // columns of a cell
  __shared__ uint32_t table[16];
  mask_selectors<ES>(table, threadIdx.x);
  wait_for_stream();
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const uint32_t rows_of_warp = 32u >> cell_shift, cell = (blockIdx.x << cell_shift) + (lane & ((1u << cell_shift) - 1u));
  const uint32_t thread_row = warp * rows_of_warp + (lane >> cell_shift);  // eight of these to a row group
  const uint32_t in_group = thread_row & 7u, step = gridDim.y * rows_of_warp;
  if (!FULL && (int64_t)cell * kCols >= K) return;
  const uint32_t chunk = ES == 2 ? cell : 2 * cell;
  const uint8_t* const meta_cell0 = meta + (!HW ? 2 * chunk
                                                : (chunk >> 3) * 2048u + 16u * in_group +
                                                      (ES == 2 ? 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) : 2u * (chunk & 7u)));
  uint32_t n = blockIdx.y * rows_of_warp + (thread_row >> 3);  // row group
  const int64_t row0 = (int64_t)n * 16 + in_group;
  const uint8_t* wp = w + row0 * row_bytes_w + (int64_t)cell * 32;
  uint8_t* yp = y + row0 * row_bytes_y + (int64_t)cell * 32;
#pragma unroll 1
  for (; n < row_groups; n += step, wp += (int64_t)step * 16 * row_bytes_w, yp += (int64_t)step * 16 * row_bytes_y) {
    uint4 in[2][2];
    bool live[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      live[h] = FULL || (int64_t)n * 16 + in_group + 8 * h < M;
      if (live[h]) ld_stream32(wp + 8 * h * row_bytes_w, in[h]);
    }
    uint32_t bits[2] = {0, 0};  // 16-bit types: in the lower half
    if constexpr (HW) {
      const uint8_t* mr = meta_cell0 + ((uint64_t)(n >> 3) * KB << 11) + 256u * (n & 7u);
      bits[0] = *reinterpret_cast<const uint32_t*>(mr);
      bits[1] = ES == 2 ? bits[0] >> 16 : *reinterpret_cast<const uint32_t*>(mr + 128);
    } else {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        if (!live[h]) continue;
        const uint16_t* mr = reinterpret_cast<const uint16_t*>(meta_cell0 + ((int64_t)n * 16 + in_group + 8 * h) * (K >> 3));
        bits[h] = mr[0];
        if (ES == 1) bits[h] |= (uint32_t)mr[1] << 16;
      }
    }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!live[h]) continue;
      uint32_t v[8] = {in[h][0].x, in[h][0].y, in[h][0].z, in[h][0].w, in[h][1].x, in[h][1].y, in[h][1].z, in[h][1].w};
#pragma unroll
      for (int g = 0; g < 8 / ES; ++g) {
        const uint32_t sel = table[(bits[h] >> (4 * g)) & 15u];
        if constexpr (ES == 2) {
          v[2 * g] = __byte_perm(v[2 * g], 0, sel & 0xFFFFu);
          v[2 * g + 1] = __byte_perm(v[2 * g + 1], 0, sel >> 16);
        } else {
          v[g] = __byte_perm(v[g], 0, sel);
        }
      }
      uint8_t* dst = yp + 8 * h * row_bytes_y;
      asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]),
                   "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
                   : "memory");
    }
  }
}

// Operands at 16-byte boundaries, and large ones.  Work unit: one 16-byte vector (two groups of a 16-bit type = one metadata byte,
// four of an 8-bit type = two bytes); launch geometry and unrolling as in prune_vec_kernel, metadata addresses as in
// compress_kernel.
// Bound by HBM.  The result is stored without an evict-first hint: it is compressed next, and as much of it as fits is then
// read from the L2 (bf16 12288 x 3072 with its compression of then 40.9 us against 42.7, device).
template <int ES, int UNROLL, bool HW>
__global__ void __launch_bounds__(kThreads) apply_mask_units_kernel(const uint8_t* w, int64_t row_bytes_w, const uint8_t* meta,
                                                                  uint8_t* y, int64_t row_bytes_y, int64_t M, int64_t K,
                                                                  int64_t KB) {
  __shared__ uint32_t table[16];
  mask_selectors<ES>(table, threadIdx.y * blockDim.x + threadIdx.x);
  wait_for_stream();
  const uint32_t units = (uint32_t)(K * ES >> 4), u0 = blockIdx.x * UNROLL * blockDim.x + threadIdx.x;
  uint32_t moff[UNROLL];  // metadata offset of this thread's units inside a row: fixed for the whole kernel
#pragma unroll
  for (int u = 0; u < UNROLL; ++u) {
    const uint32_t unit = u0 + u * blockDim.x, chunk = ES == 2 ? unit >> 1 : unit;
    moff[u] = !HW ? unit * (2 / ES)
                  : (chunk >> 3) * 2048u + (ES == 2 ? 128u * (chunk & 1u) + 4u * ((chunk >> 1) & 3u) + (unit & 1u) : 2u * (chunk & 7u));
  }
  for (int64_t row = (int64_t)blockIdx.y * blockDim.y + threadIdx.y; row < M; row += (int64_t)gridDim.y * blockDim.y) {
    const uint32_t r = (uint32_t)row & 127u;
    const uint8_t* mr = HW ? meta + (row >> 7) * (KB * 2048) + (ES == 2 ? 16u * (r & 7u) + 2u * ((r >> 3) & 1u) + 256u * (r >> 4) : 16u * r)
                           : meta + row * (K >> 3);
    const uint8_t* wr = w + row * row_bytes_w;
    uint8_t* yr = y + row * row_bytes_y;
    uint4 in[UNROLL];
    uint32_t bits[UNROLL];
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t unit = u0 + u * blockDim.x;
      if (unit < units) {
        in[u] = __ldcs(reinterpret_cast<const uint4*>(wr + unit * 16u));
        bits[u] = ES == 2 ? *(mr + moff[u]) : *reinterpret_cast<const uint16_t*>(mr + moff[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < UNROLL; ++u) {
      const uint32_t unit = u0 + u * blockDim.x;
      if (unit >= units) continue;
      const uint4 v = in[u];
      uint4 o;
      if (ES == 2) {
        const uint32_t s0 = table[bits[u] & 15u], s1 = table[bits[u] >> 4];
        o = make_uint4(__byte_perm(v.x, 0, s0 & 0xFFFFu), __byte_perm(v.y, 0, s0 >> 16), __byte_perm(v.z, 0, s1 & 0xFFFFu),
                       __byte_perm(v.w, 0, s1 >> 16));
      } else {
        o = make_uint4(__byte_perm(v.x, 0, table[bits[u] & 15u]), __byte_perm(v.y, 0, table[(bits[u] >> 4) & 15u]),
                       __byte_perm(v.z, 0, table[(bits[u] >> 8) & 15u]), __byte_perm(v.w, 0, table[bits[u] >> 12]));
      }
      *reinterpret_cast<uint4*>(yr + unit * 16u) = o;
    }
  }
}

// One thread per 8 columns (two groups = one metadata byte in either layout).
template <typename T>
__global__ void __launch_bounds__(kThreads) apply_mask_kernel(const T* __restrict__ w, int64_t ldw, const uint8_t* meta,
                                                              int layout, T* y, int64_t ldy, int64_t M, int64_t K,
                                                              int64_t KB) {
  constexpr int ES = sizeof(T);
  const int64_t bytes = K >> 3;
  const int64_t id = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (id >= M * bytes) return;
  const int64_t row = id / bytes, bi = id - row * bytes;
  int64_t off;
  if (layout == SP24_META_CANONICAL) {
    off = row * bytes + bi;
  } else {
    const int64_t chunk = bi >> 1, blk = (row >> 7) * KB + (chunk >> 3);
    const int r = (int)(row & 127), cl = (int)(chunk & 7);
    const int in_blk = ES == 2 ? 16 * (r & 7) + 2 * ((r >> 3) & 1) + 256 * (r >> 4) + 128 * (cl & 1) + 4 * (cl >> 1)
                               : 16 * r + 2 * cl;
    off = blk * 2048 + in_blk + (bi & 1);
  }
  const uint32_t mbyte = meta[off];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t nib = (mbyte >> (4 * h)) & 0xFu, p0 = nib & 3u, p1 = nib >> 2;
    const T* src = w + row * ldw + 8 * bi + 4 * h;
    T* dst = y + row * ldy + 8 * bi + 4 * h;
    T e[4];
#pragma unroll
    for (int p = 0; p < 4; ++p) e[p] = src[p];
#pragma unroll
    for (int p = 0; p < 4; ++p) dst[p] = ((uint32_t)p == p0 || (uint32_t)p == p1) ? e[p] : (T)0;
  }
}

// ---- 2:4 along rows and columns ------------------------------------------------------------------------
// The 90 patterns: every row keeps one of the six pairs {01,02,03,12,13,23} (in that order, index 0..5)
// and every column ends up with exactly two kept entries.  Patterns are numbered in lexicographic order
// of their four row indices; entry n packs the four 3-bit row indices of pattern n.  The table is built
// at compile time so that the search below unrolls into straight-line code on registers.
struct PatternTable {
  uint16_t v[90];
};
constexpr uint32_t pair_mask(int q) { return q == 0 ? 0x3u : q == 1 ? 0x5u : q == 2 ? 0x9u : q == 3 ? 0x6u : q == 4 ? 0xAu : 0xCu; }
constexpr PatternTable make_patterns() {
  PatternTable t{};
  int n = 0;
  for (int a = 0; a < 6; ++a)
    for (int b = 0; b < 6; ++b)
      for (int c = 0; c < 6; ++c)
        for (int d = 0; d < 6; ++d) {
          bool ok = true;
          for (int col = 0; col < 4; ++col) {
            const uint32_t cnt = ((pair_mask(a) >> col) & 1u) + ((pair_mask(b) >> col) & 1u) +
                                 ((pair_mask(c) >> col) & 1u) + ((pair_mask(d) >> col) & 1u);
            ok = ok && cnt == 2u;
          }
          if (ok && n < 90) t.v[n++] = (uint16_t)(a | (b << 3) | (c << 6) | (d << 9));
        }
  return t;
}
constexpr PatternTable kPatternTable = make_patterns();
static_assert(kPatternTable.v[89] != 0 && kPatternTable.v[0] == (0 | (0 << 3) | (5 << 6) | (5 << 9)),
              "90 patterns, the first keeps columns 0,1 in rows 0,1 and 2,3 in rows 2,3");

template <int N>
struct PatternSearch {
  // patterns N..89 in order; `s[i][q]`: kept magnitude of row i under pair q
  static __device__ __forceinline__ void run(const float (&s)[4][6], float& best, uint32_t& best_pat) {
    constexpr uint32_t pat = kPatternTable.v[N];
    const float sc = __fadd_rn(__fadd_rn(__fadd_rn(s[0][pat & 7u], s[1][(pat >> 3) & 7u]), s[2][(pat >> 6) & 7u]),
                               s[3][(pat >> 9) & 7u]);
    if (sc > best) { best = sc; best_pat = pat; }
    PatternSearch<N + 1>::run(s, best, best_pat);
  }
};
template <>
struct PatternSearch<90> {
  static __device__ __forceinline__ void run(const float (&)[4][6], float&, uint32_t&) {}
};

// Score of a pattern: ((s0 + s1) + s2) + s3 with s_i = |x[i, c]| + |x[i, c']| (c < c'), all in FP32 (exact
// for int8); the first pattern with the largest score wins.  One thread per 4 x 4 block.
template <int DT, typename T>
__global__ void __launch_bounds__(kThreads) prune_2d_kernel(const T* __restrict__ x, int64_t ldx, T* y, int64_t ldy,
                                                            int64_t block_rows, int64_t block_cols) {
  const int64_t bc = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (bc >= block_cols) return;
  for (int64_t br = blockIdx.y; br < block_rows; br += gridDim.y) {
    T e[4][4];
    float s[4][6];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const T* src = x + (4 * br + i) * ldx + 4 * bc;
      if (sizeof(T) == 2 && ((reinterpret_cast<uintptr_t>(src) & 7u) == 0)) {
        const uint2 v = *reinterpret_cast<const uint2*>(src);
        e[i][0] = (T)(v.x & 0xFFFFu); e[i][1] = (T)(v.x >> 16); e[i][2] = (T)(v.y & 0xFFFFu); e[i][3] = (T)(v.y >> 16);
      } else if (sizeof(T) == 1 && ((reinterpret_cast<uintptr_t>(src) & 3u) == 0)) {
        const uint32_t v = *reinterpret_cast<const uint32_t*>(src);
        e[i][0] = (T)(v & 0xFFu); e[i][1] = (T)((v >> 8) & 0xFFu); e[i][2] = (T)((v >> 16) & 0xFFu); e[i][3] = (T)(v >> 24);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) e[i][j] = src[j];
      }
      float a[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = magnitude_of<DT>(e[i][j]);
      s[i][0] = __fadd_rn(a[0], a[1]); s[i][1] = __fadd_rn(a[0], a[2]); s[i][2] = __fadd_rn(a[0], a[3]);
      s[i][3] = __fadd_rn(a[1], a[2]); s[i][4] = __fadd_rn(a[1], a[3]); s[i][5] = __fadd_rn(a[2], a[3]);
    }
    float best = -1.f;
    uint32_t best_pat = 0;
    PatternSearch<0>::run(s, best, best_pat);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t q = (best_pat >> (3 * i)) & 7u;
      const uint32_t m = q == 0 ? 0x3u : q == 1 ? 0x5u : q == 2 ? 0x9u : q == 3 ? 0x6u : q == 4 ? 0xAu : 0xCu;
      T* dst = y + (4 * br + i) * ldy + 4 * bc;
      T o[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) o[j] = ((m >> j) & 1u) ? e[i][j] : (T)0;
      if (sizeof(T) == 2 && ((reinterpret_cast<uintptr_t>(dst) & 7u) == 0)) {
        *reinterpret_cast<uint2*>(dst) = make_uint2((uint32_t)(uint16_t)o[0] | ((uint32_t)(uint16_t)o[1] << 16),
                                                     (uint32_t)(uint16_t)o[2] | ((uint32_t)(uint16_t)o[3] << 16));
      } else if (sizeof(T) == 1 && ((reinterpret_cast<uintptr_t>(dst) & 3u) == 0)) {
        *reinterpret_cast<uint32_t*>(dst) = (uint32_t)(uint8_t)o[0] | ((uint32_t)(uint8_t)o[1] << 8) |
                                            ((uint32_t)(uint8_t)o[2] << 16) | ((uint32_t)(uint8_t)o[3] << 24);
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j) dst[j] = o[j];
      }
    }
  }
}

}  // namespace
}  // namespace sp24

using namespace sp24;

extern "C" sp24_status sp24_kept_magnitude(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx,
                                           const int32_t* perm, double* result, void* stream) {
  SP24_RETURN_IF(!is_ab_type(t) || is_fp8(t), SP24_ERR_DTYPE);
  SP24_RETURN_IF(M < 0 || K < 0 || K % 4 != 0, SP24_ERR_SHAPE);
  SP24_RETURN_IF(result == nullptr, SP24_ERR_NULL);
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(x == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldx < K, SP24_ERR_STRIDE);
  sp24_status st = check_arch();
  if (st != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int es = elem_bytes(t);
  const bool rows_aligned = aligned16(x) && (ldx * es) % 16 == 0 && (K * es) % 16 == 0;
  if (rows_aligned && perm == nullptr) {
    const int64_t vpr = K * es / 16;
    dim3 grid((unsigned)((vpr + kThreads - 1) / kThreads), (unsigned)(M < 4096 ? M : 4096), 1);
    const uint8_t* xb = static_cast<const uint8_t*>(x);
    if (t == SP24_F16) kept_magnitude_vec_kernel<0><<<grid, kThreads, 0, s>>>(xb, ldx * es, M, vpr, result);
    else if (t == SP24_BF16) kept_magnitude_vec_kernel<1><<<grid, kThreads, 0, s>>>(xb, ldx * es, M, vpr, result);
    else kept_magnitude_vec_kernel<2><<<grid, kThreads, 0, s>>>(xb, ldx * es, M, vpr, result);
    return cuda_status(cudaGetLastError());
  }
  if (rows_aligned && aligned16(perm) && K * es <= 48 * 1024) {
    const unsigned grid = (unsigned)(M < 148 * 8 ? M : 148 * 8);
    const size_t smem = (size_t)K * es;
    const uint8_t* xb = static_cast<const uint8_t*>(x);
    if (t == SP24_F16)
      kept_magnitude_perm_kernel<0, uint16_t><<<grid, kThreads, smem, s>>>(xb, ldx * es, M, K, perm, result);
    else if (t == SP24_BF16)
      kept_magnitude_perm_kernel<1, uint16_t><<<grid, kThreads, smem, s>>>(xb, ldx * es, M, K, perm, result);
    else
      kept_magnitude_perm_kernel<2, int8_t><<<grid, kThreads, smem, s>>>(xb, ldx * es, M, K, perm, result);
    return cuda_status(cudaGetLastError());
  }
  const int64_t groups = K / 4, total = M * groups;
  int64_t blocks = (total + kThreads - 1) / kThreads;
  if (blocks > 148 * 16) blocks = 148 * 16;
  if (t == SP24_F16)
    kept_magnitude_kernel<0, uint16_t><<<(unsigned)blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, M, groups, perm, result);
  else if (t == SP24_BF16)
    kept_magnitude_kernel<1, uint16_t><<<(unsigned)blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, M, groups, perm, result);
  else
    kept_magnitude_kernel<2, int8_t><<<(unsigned)blocks, kThreads, 0, s>>>((const int8_t*)x, ldx, M, groups, perm, result);
  return cuda_status(cudaGetLastError());
}

extern "C" sp24_status sp24_apply_mask(sp24_dtype t, int64_t M, int64_t K, const void* w, int64_t ldw, const void* meta,
                                       sp24_meta_layout l, void* y, int64_t ldy, void* stream) {
  SP24_RETURN_IF(!is_ab_type(t), SP24_ERR_DTYPE);
  SP24_RETURN_IF(M < 0 || K < 0 || K % 8 != 0, SP24_ERR_SHAPE);
  SP24_RETURN_IF(l != SP24_META_CANONICAL && l != SP24_META_TCGEN05, SP24_ERR_UNSUPPORTED);
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(w == nullptr || meta == nullptr || y == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldw < K || ldy < K, SP24_ERR_STRIDE);
  sp24_status st = check_arch();
  if (st != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t total = M * (K / 8), KB = 2 * ((K + 255) / 256);
  const int es = elem_bytes(t);
  if (K % 16 == 0 && aligned16(w) && aligned16(y) && aligned16(meta) && (ldw * es) % 16 == 0 && (ldy * es) % 16 == 0 &&
      row_offsets_fit(K, es, l)) {
    const bool hw = l == SP24_META_TCGEN05;
    const int64_t cols = es == 2 ? 16 : 32, cells = K / cols;
    auto by32 = [&](const void* p, int64_t ld) { return reinterpret_cast<uintptr_t>(p) % 32 == 0 && ld * es % 32 == 0; };
    constexpr int UNROLL = 4;
    const RowLaunch L(K * es / 16, M, UNROLL);
    // Whole cells of a matrix beyond 80 MiB go by units as well, unless these leave three of ten lanes idle: HBM bounds both, and a
    // warp's units are 512 bytes of one row.  Us, device, units and cells, alone and with the compression: bf16 53517 x 3248 107.3,
    // 111.4, 193.3, 197.0; 16801 x 14736 152.2, 155.0, 275.1, 277.9; 49152 x 12288 362.5, 362.5, 641, 641; int8 306380 x 1568 153.6,
    // 162.8, 327, 336; below the line bf16 6172 x 5424 (67 MB) 18.2, 17.5, 33.6, 33.6, int8
    // 9740 x 7424 (72 MB) 22.9, 21.5, 44.9, 43.8.
    const bool large = M * K * es > (int64_t)80 << 20 && 10 * (K * es / 16) >= 7 * (int64_t)L.grid.x * L.block.x * UNROLL;
    if (K % cols == 0 && by32(w, ldw) && by32(y, ldy) && !large) {
      // Cells of a row to a warp: 32, 16 or 8, the most of which few lanes are idle (32 and fewer, us, with the compression: bf16
      // 49152 x 256 15.3, 13.5; 6088 x 11632, whose 727 cells are whole only by 8, 77.4, 78.3).
      auto padded = [&](int log) { return (cells + (1 << log) - 1) >> log << log; };
      const int64_t most = padded(3) + cells / 16;
      const int shift = padded(5) <= most ? 5 : padded(4) <= most ? 4 : 3;
      const int64_t units = padded(shift) >> shift, groups = (M + 15) / 16, per_block = 32 >> shift;
      int64_t steps = (groups + per_block - 1) / per_block;
      if (steps > 32768) steps = 32768;
      const bool full = M % 16 == 0 && cells == units << shift;
      auto launch = [&](auto kernel) {
        return launch_streaming(kernel, dim3((unsigned)units, (unsigned)steps, 1), dim3(kThreads), s, (const uint8_t*)w, ldw * es,
                                (const uint8_t*)meta, (uint8_t*)y, ldy * es, M, K, (uint32_t)groups, (uint32_t)KB, shift);
      };
      if (es == 2 && full) return hw ? launch(Kernel<apply_mask_vec_kernel<2, true, true>>{}) : launch(Kernel<apply_mask_vec_kernel<2, false, true>>{});
      if (es == 2) return hw ? launch(Kernel<apply_mask_vec_kernel<2, true, false>>{}) : launch(Kernel<apply_mask_vec_kernel<2, false, false>>{});
      if (full) return hw ? launch(Kernel<apply_mask_vec_kernel<1, true, true>>{}) : launch(Kernel<apply_mask_vec_kernel<1, false, true>>{});
      return hw ? launch(Kernel<apply_mask_vec_kernel<1, true, false>>{}) : launch(Kernel<apply_mask_vec_kernel<1, false, false>>{});
    }
    auto launch = [&](auto kernel) {
      return launch_streaming(kernel, L.grid, L.block, s, (const uint8_t*)w, ldw * es, (const uint8_t*)meta, (uint8_t*)y, ldy * es, M, K, KB);
    };
    if (es == 2) return hw ? launch(Kernel<apply_mask_units_kernel<2, UNROLL, true>>{}) : launch(Kernel<apply_mask_units_kernel<2, UNROLL, false>>{});
    return hw ? launch(Kernel<apply_mask_units_kernel<1, UNROLL, true>>{}) : launch(Kernel<apply_mask_units_kernel<1, UNROLL, false>>{});
  }
  const unsigned blocks = (unsigned)((total + kThreads - 1) / kThreads);
  if (elem_bytes(t) == 2)
    apply_mask_kernel<uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)w, ldw, (const uint8_t*)meta, (int)l,
                                                            (uint16_t*)y, ldy, M, K, KB);
  else
    apply_mask_kernel<int8_t><<<blocks, kThreads, 0, s>>>((const int8_t*)w, ldw, (const uint8_t*)meta, (int)l, (int8_t*)y,
                                                          ldy, M, K, KB);
  return cuda_status(cudaGetLastError());
}

extern "C" sp24_status sp24_prune_2d(sp24_dtype t, int64_t M, int64_t K, const void* x, int64_t ldx, void* y, int64_t ldy,
                                     void* stream) {
  SP24_RETURN_IF(!is_ab_type(t) || is_fp8(t), SP24_ERR_DTYPE);
  SP24_RETURN_IF(M < 0 || K < 0 || K % 4 != 0 || M % 4 != 0, SP24_ERR_SHAPE);
  if (M == 0 || K == 0) return SP24_OK;
  SP24_RETURN_IF(x == nullptr || y == nullptr, SP24_ERR_NULL);
  SP24_RETURN_IF(ldx < K || ldy < K, SP24_ERR_STRIDE);
  sp24_status st = check_arch();
  if (st != SP24_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const int64_t br = M / 4, bc = K / 4;
  const dim3 blocks((unsigned)((bc + kThreads - 1) / kThreads), (unsigned)(br < 16384 ? br : 16384), 1);
  if (t == SP24_F16)
    prune_2d_kernel<0, uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, (uint16_t*)y, ldy, br, bc);
  else if (t == SP24_BF16)
    prune_2d_kernel<1, uint16_t><<<blocks, kThreads, 0, s>>>((const uint16_t*)x, ldx, (uint16_t*)y, ldy, br, bc);
  else
    prune_2d_kernel<2, int8_t><<<blocks, kThreads, 0, s>>>((const int8_t*)x, ldx, (int8_t*)y, ldy, br, bc);
  return cuda_status(cudaGetLastError());
}
