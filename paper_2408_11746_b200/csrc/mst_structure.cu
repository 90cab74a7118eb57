// Sparse structure of a layer: bit mask -> CSR (+ CSC view) by popcount, exclusive prefix scan and fill.
//
// The mask is kept as 32-bit words, wpr words per row.  Because canonical CSR order (rows ascending,
// columns ascending) is the order of the flat index o*I+i, the CSR position of an entry is the number of
// set bits before it: an exclusive scan of the per-word popcounts plus a popcount inside the word.
// The same holds for the CSC view on the transposed bit mask.  Everything below is integer work,
// stream-ordered, with no inter-block waiting (the scan is three plain kernels).
#include "mst_internal.cuh"
#include "mst_tc_gemm.cuh"
#include "mst_bits.cuh"

#include <cuda_bf16.h>

namespace {

constexpr int SCAN_THREADS = 256;
constexpr int SCAN_ITEMS = 8;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_ITEMS;

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

// ---- exclusive scan of int32, n up to 2^31: out[0..n], out[n] = total -------------------------
__device__ int block_reduce_sum(int v, int* sh) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  int r = 0;
  if (threadIdx.x < 32) {
    r = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0;
    for (int o = 16; o; o >>= 1) r += __shfl_xor_sync(0xffffffffu, r, o);
  }
  __syncthreads();
  return r;  // valid in warp 0
}

__global__ void scan_tile_sums(const int32_t* __restrict__ in, int64_t n, int32_t* __restrict__ sums,
                               const int* __restrict__ enabled) {
  __shared__ int sh[32];
  if (enabled && !*enabled) return;
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE;
  int v = 0;
  for (int j = 0; j < SCAN_ITEMS; ++j) {
    const int64_t i = base + (int64_t)j * SCAN_THREADS + threadIdx.x;
    if (i < n) v += in[i];
  }
  const int r = block_reduce_sum(v, sh);
  if (threadIdx.x == 0) sums[blockIdx.x] = r;
}

// one block: in-place exclusive scan of the tile sums (m values)
__global__ void scan_sums_inplace(int32_t* sums, int64_t m, const int* __restrict__ enabled) {
  __shared__ int sh[32];
  __shared__ int carry;
  if (enabled && !*enabled) return;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int64_t base = 0; base < m; base += blockDim.x) {
    const int64_t i = base + threadIdx.x;
    const int v = i < m ? sums[i] : 0;
    int x = v;  // inclusive scan inside the warp
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, x, o);
      if ((threadIdx.x & 31) >= o) x += y;
    }
    if ((threadIdx.x & 31) == 31) sh[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x < 32) {
      int w = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : 0;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, w, o);
        if (threadIdx.x >= o) w += y;
      }
      sh[threadIdx.x] = w;  // inclusive over warps
    }
    __syncthreads();
    const int warp_off = (threadIdx.x >> 5) ? sh[(threadIdx.x >> 5) - 1] : 0;
    const int c = carry;
    if (i < m) sums[i] = c + warp_off + x - v;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = c + warp_off + x;
    __syncthreads();
  }
}

__global__ void scan_tiles(const int32_t* __restrict__ in, int64_t n, const int32_t* __restrict__ sums,
                           int32_t* __restrict__ out, const int* __restrict__ enabled) {
  // thread owns SCAN_ITEMS consecutive elements
  __shared__ int sh[32];
  if (enabled && !*enabled) return;
  const int64_t base = (int64_t)blockIdx.x * SCAN_TILE + (int64_t)threadIdx.x * SCAN_ITEMS;
  int v[SCAN_ITEMS];
  int t = 0;
  for (int j = 0; j < SCAN_ITEMS; ++j) {
    v[j] = (base + j < n) ? in[base + j] : 0;
    t += v[j];
  }
  int x = t;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if ((threadIdx.x & 31) >= o) x += y;
  }
  if ((threadIdx.x & 31) == 31) sh[threadIdx.x >> 5] = x;
  __syncthreads();
  if (threadIdx.x < 32) {
    int w = threadIdx.x < (SCAN_THREADS >> 5) ? sh[threadIdx.x] : 0;
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (threadIdx.x >= o) w += y;
    }
    sh[threadIdx.x] = w;
  }
  __syncthreads();
  int run = sums[blockIdx.x] + ((threadIdx.x >> 5) ? sh[(threadIdx.x >> 5) - 1] : 0) + x - t;
  for (int j = 0; j < SCAN_ITEMS; ++j) {
    if (base + j < n) out[base + j] = run;
    run += v[j];
    if (base + j == n - 1) out[n] = run;
  }
}

__global__ void scan_empty(int32_t* out) { out[0] = 0; }

// ---- pack: byte mask -> bit mask -> CSR in two launches ----------------------------------------------------------------------
// Launch 1 turns 256 mask words per block into bits and leaves the block's entry count; launch 2 adds up the counts of the
// blocks before its own (of many blocks: reads their scan), scans its words and writes their part of the structure, one warp per word (lane = bit: reads of
// W and writes of the compacted arrays are coalesced), eight words in flight, or half a word per thread where there are few entries.
// 4096 x 1024 bf16, d = 0.1, with its export: 31 us with whole words only (a warp instruction per word and array, a tenth of its lanes at
// work), 24 us with half words; separate bits, popcounts, three-kernel scans (twice) and one-word-per-warp fill, eleven launches, 106 us.
constexpr int PACK_THREADS = 256;
constexpr int PACK_WORDS = PACK_THREADS;       // mask words per block

__device__ __forceinline__ uint32_t nibble_of(uint32_t four_bytes) {   // bit j: byte j is not zero
  const uint32_t m = __vcmpne4(four_bytes, 0u) & 0x01010101u;
  return (m * 0x01020408u) >> 24;
}

__global__ void __launch_bounds__(PACK_THREADS) pack_bits_kernel(const uint8_t* __restrict__ mask, int O, int I, int wpr, int vec,
                                                                 uint32_t* __restrict__ bits, int32_t* __restrict__ sums) {
  __shared__ int sh[32];
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int64_t nwords = (int64_t)O * wpr, w0 = (int64_t)blockIdx.x * PACK_WORDS;
  int count = 0;
  if (vec) {   // mask words tile the bytes (I a multiple of 32) and start on 16-byte boundaries
    {
      const int64_t w = w0 + threadIdx.x;
      if (w < nwords) {
        const uint4* src = reinterpret_cast<const uint4*>(mask + w * 32);
        const uint4 a = __ldg(src), b = __ldg(src + 1);
        const uint32_t word = nibble_of(a.x) | (nibble_of(a.y) << 4) | (nibble_of(a.z) << 8) | (nibble_of(a.w) << 12) |
                              (nibble_of(b.x) << 16) | (nibble_of(b.y) << 20) | (nibble_of(b.z) << 24) | (nibble_of(b.w) << 28);
        bits[w] = word;
        count += __popc(word);
      }
    }
  } else {     // a warp takes 32 neighbouring words, lane = column; lane k keeps word k
    const int lane = threadIdx.x & 31;
    const int64_t wb = w0 + (threadIdx.x >> 5) * 32;
    if (wb < nwords) {
      uint32_t mine = 0;
      int o = (int)(wb / wpr), wc = (int)(wb - (int64_t)o * wpr);
#pragma unroll 8
      for (int k = 0; k < 32; ++k) {
        const int c = wc * 32 + lane;
        const bool on = wb + k < nwords && c < I && mask[(int64_t)o * I + c] != 0;
        const uint32_t word = __ballot_sync(0xffffffffu, on);
        if (lane == k) mine = word;
        if (++wc == wpr) { wc = 0; ++o; }
      }
      if (wb + lane < nwords) {
        bits[wb + lane] = mine;
        count += __popc(mine);
      }
    }
  }
  const int r = block_reduce_sum(count, sh);
  if (threadIdx.x == 0) sums[blockIdx.x] = r;
}

// sums: the blocks' counts, or with `scanned` the counts before each of them.  Entries at positions >= cap are counted but not written.  *total receives the number of entries (device memory or mapped host
// memory); wscan may be NULL.
template <typename V, typename COL>
__global__ void __launch_bounds__(PACK_THREADS) pack_fill_kernel(const uint32_t* __restrict__ bits, const int32_t* __restrict__ sums, int scanned, int O,
                                                                 int wpr, const V* __restrict__ W, int64_t ldw, int64_t cap,
                                                                 int32_t* __restrict__ wscan, int32_t* __restrict__ row_ptr,
                                                                 COL* __restrict__ col_idx, V* __restrict__ vals, volatile int32_t* total) {
  __shared__ int sh[32];
  __shared__ int before_sh;
  __shared__ uint32_t word_sh[PACK_WORDS];
  __shared__ int32_t at_sh[PACK_WORDS];
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int64_t nwords = (int64_t)O * wpr, w0 = (int64_t)blockIdx.x * PACK_WORDS;
  int before = 0;
  if (scanned) {
    before = sums[blockIdx.x];
  } else {
    for (int j = threadIdx.x; j < (int)blockIdx.x; j += PACK_THREADS) before += sums[j];
    before = block_reduce_sum(before, sh);
  }
  if (threadIdx.x == 0) before_sh = before;
  const int64_t my_w = w0 + threadIdx.x;
  const uint32_t my_bits = my_w < nwords ? bits[my_w] : 0u;
  const int mine = __popc(my_bits);
  int incl = mine;
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if ((threadIdx.x & 31) >= o) incl += y;
  }
  __syncthreads();   // sh is free, before_sh is set
  if ((threadIdx.x & 31) == 31) sh[threadIdx.x >> 5] = incl;
  __syncthreads();
  int at = before_sh + incl - mine;
  for (int k = 0; k < (int)(threadIdx.x >> 5); ++k) at += sh[k];
  word_sh[threadIdx.x] = my_bits;
  at_sh[threadIdx.x] = at;
  if (my_w < nwords) {
    if (wscan) wscan[my_w] = at;
    const unsigned o = (unsigned)my_w / (unsigned)wpr;
    if (o * (unsigned)wpr == (unsigned)my_w) row_ptr[o] = at;
    if (my_w == nwords - 1) {
      at += mine;
      if (wscan) wscan[nwords] = at;
      row_ptr[O] = at;
      if (total) *total = at;
    }
  }
  // Few entries: half a word per thread, four entries at a time; a store then touches many lines, but there are few stores.
  if (__syncthreads_count(mine > 8) < PACK_THREADS / 8) {
    for (int i = threadIdx.x; i < 2 * PACK_WORDS; i += PACK_THREADS) {
      const int li = i >> 1;
      const uint32_t word = word_sh[li];
      uint32_t m = (i & 1) ? word & 0xFFFF0000u : word & 0xFFFFu;
      if (m == 0u) continue;
      const unsigned w = (unsigned)(w0 + li), o = w / (unsigned)wpr;
      const int c0 = (int)(w - o * (unsigned)wpr) * 32;
      const V* src = W + (int64_t)o * ldw + c0;
      int64_t pos = (int64_t)at_sh[li] + ((i & 1) ? __popc(word & 0xFFFFu) : 0);
      while (m) {
        int b[4];
        V v[4];
        const int n = __popc(m);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          b[j] = m ? __ffs(m) - 1 : 0;
          m &= m - 1u;
          v[j] = src[b[j]];   // without an entry column 0 of the word, inside the row
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          if (j < n && pos + j < cap) {
            col_idx[pos + j] = (COL)(c0 + b[j]);
            vals[pos + j] = v[j];
          }
        }
        pos += 4;
      }
    }
    return;
  }
  const int lane = threadIdx.x & 31;
  constexpr int U = 8;
  for (int l0 = threadIdx.x >> 5; l0 < PACK_WORDS; l0 += (PACK_THREADS / 32) * U) {
    V v[U];
    int64_t pos[U];
    int col[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int li = l0 + u * (PACK_THREADS / 32);
      const uint32_t word = word_sh[li];   // 0 beyond the last word
      const unsigned w = (unsigned)(w0 + li), o = w / (unsigned)wpr;
      pos[u] = ((word >> lane) & 1u) ? (int64_t)at_sh[li] + __popc(word & lanemask_lt()) : cap;
      col[u] = (int)(w - o * (unsigned)wpr) * 32 + lane;
      if (pos[u] < cap) v[u] = W[(int64_t)o * ldw + col[u]];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (pos[u] < cap) {
        col_idx[pos[u]] = (COL)col[u];
        vals[pos[u]] = v[u];
      }
    }
  }
}

__global__ void popc_words(const uint32_t* __restrict__ bits, int64_t n, int32_t* __restrict__ cnt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) cnt[i] = __popc(bits[i]);
}

// new = (old & ~pruned) | grad | rand
__global__ void combine_bits(const uint32_t* __restrict__ oldb, const uint32_t* __restrict__ pruned,
                             const uint32_t* __restrict__ grad, const uint32_t* __restrict__ rnd, int64_t n,
                             uint32_t* __restrict__ out, int32_t* __restrict__ cnt) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const uint32_t b = (oldb[i] & ~pruned[i]) | grad[i] | rnd[i];
    out[i] = b;
    cnt[i] = __popc(b);
  }
}

// ---- CSR fill: one warp per word, lane = bit ---------------------------------------------------
// Source of a value: dense W (pack) or the previous structure (update: survivors keep their value, others +0).
template <typename V>
__global__ void fill_csr(const uint32_t* __restrict__ bits, const int32_t* __restrict__ wscan, int O, int I, int wpr,
                         uint16_t* __restrict__ col_idx, V* __restrict__ vals, int32_t* __restrict__ row_ptr,
                         const V* __restrict__ dense_W, int64_t ldw, const uint32_t* __restrict__ old_bits,
                         const int32_t* __restrict__ old_wscan, const V* __restrict__ old_vals) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= (int64_t)O * wpr) return;
  mst_fill_csr_word<V>(w, threadIdx.x & 31, bits, wscan, O, I, wpr, col_idx, vals, row_ptr, dense_W, ldw, old_bits,
                       old_wscan, old_vals);
}

// ---- bit transpose: one warp per 32x32 bit tile -------------------------------------------------
__global__ void transpose_bits(const uint32_t* __restrict__ bits, int O, int I, int wpr, int wpc,
                               uint32_t* __restrict__ bitsT) {
  const int64_t tile = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (tile >= (int64_t)wpc * wpr) return;
  mst_transpose_tile(tile, threadIdx.x & 31, bits, O, I, wpr, wpc, bitsT);
}

__global__ void fill_csc(const uint32_t* __restrict__ bitsT, const int32_t* __restrict__ wscanT, int O, int I, int wpr,
                         int wpc, const uint32_t* __restrict__ bits, const int32_t* __restrict__ wscan,
                         uint16_t* __restrict__ row_idx, int32_t* __restrict__ perm, int32_t* __restrict__ col_ptr) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= (int64_t)I * wpc) return;
  mst_fill_csc_word(w, threadIdx.x & 31, bitsT, wscanT, O, I, wpr, wpc, bits, wscan, row_idx, perm, col_ptr);
}

// ---- export / validate ---------------------------------------------------------------------------
// row pointers, column indices (widened) and values of the live structure in one launch; any destination may be NULL
template <typename V>
__global__ void __launch_bounds__(256) export_kernel(const int32_t* __restrict__ ptr, int n_ptr, const uint16_t* __restrict__ idx,
                                                     const V* __restrict__ vals, int64_t nnz, int32_t* __restrict__ ptr_out,
                                                     int32_t* __restrict__ idx_out, V* __restrict__ vals_out, int vec) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, threads = (int64_t)gridDim.x * blockDim.x;
  if (ptr_out)
    for (int64_t i = t; i < n_ptr; i += threads) ptr_out[i] = ptr[i];
  for (int64_t i = 4 * t; i < nnz; i += 4 * threads) {   // the stored arrays start on 256-byte boundaries
    const int n = nnz - i < 4 ? (int)(nnz - i) : 4;
    if (idx_out) {
      if (vec && n == 4) {
        const ushort4 c = *reinterpret_cast<const ushort4*>(idx + i);
        *reinterpret_cast<int4*>(idx_out + i) = make_int4(c.x, c.y, c.z, c.w);
      } else {
        for (int j = 0; j < n; ++j) idx_out[i + j] = idx[i + j];
      }
    }
    if (vals_out) {
      if (vec && n == 4) {
        if (sizeof(V) == 4) *reinterpret_cast<uint4*>(vals_out + i) = *reinterpret_cast<const uint4*>(vals + i);
        else *reinterpret_cast<uint2*>(vals_out + i) = *reinterpret_cast<const uint2*>(vals + i);
      } else {
        for (int j = 0; j < n; ++j) vals_out[i + j] = vals[i + j];
      }
    }
  }
}

__global__ void validate_rows(const int32_t* __restrict__ row_ptr, const uint16_t* __restrict__ col_idx,
                              const uint32_t* __restrict__ bits, int O, int I, int wpr, int64_t nnz,
                              int32_t* __restrict__ flags) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o >= O) return;
  bool bad = false;
  const int32_t a = row_ptr[o], b = row_ptr[o + 1];
  if (o == 0 && a != 0) bad = true;
  if (o == O - 1 && b != nnz) bad = true;
  if (a > b || a < 0 || b > nnz) {
    bad = true;
  } else {
    int prev = -1, pc = 0;
    for (int32_t k = a; k < b; ++k) {
      const int c = col_idx[k];
      if (c <= prev || c >= I) { bad = true; break; }
      if (!((bits[(int64_t)o * wpr + (c >> 5)] >> (c & 31)) & 1u)) { bad = true; break; }
      prev = c;
    }
    for (int w = 0; w < wpr; ++w) pc += __popc(bits[(int64_t)o * wpr + w]);
    if (pc != b - a) bad = true;
  }
  if (bad) atomicOr(&flags[0], MST_FLAG_CORRUPT);
}

__global__ void validate_cols(const int32_t* __restrict__ col_ptr, const uint16_t* __restrict__ row_idx,
                              const int32_t* __restrict__ perm, const int32_t* __restrict__ row_ptr,
                              const uint16_t* __restrict__ col_idx, int O, int I, int64_t nnz,
                              int32_t* __restrict__ flags) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= I) return;
  bool bad = false;
  const int32_t a = col_ptr[i], b = col_ptr[i + 1];
  if (i == 0 && a != 0) bad = true;
  if (i == I - 1 && b != nnz) bad = true;
  if (a > b || a < 0 || b > nnz) {
    bad = true;
  } else {
    int prev = -1;
    for (int32_t k = a; k < b; ++k) {
      const int o = row_idx[k];
      const int32_t p = perm[k];
      if (o <= prev || o >= O || p < 0 || p >= nnz) { bad = true; break; }
      if (p < row_ptr[o] || p >= row_ptr[o + 1] || col_idx[p] != i) { bad = true; break; }
      prev = o;
    }
  }
  if (bad) atomicOr(&flags[0], MST_FLAG_CORRUPT);
}

inline unsigned blocks_for(int64_t n, int per_block) { return (unsigned)((n + per_block - 1) / per_block); }

}  // namespace

int64_t mst_scan_block_sums_len(int64_t n) { return (n + SCAN_TILE - 1) / SCAN_TILE + 1 + 1024; }

mst_status_t mst_scan_i32_if(const int32_t* in, int32_t* out, int64_t n, int32_t* block_sums, const int* enabled,
                             cudaStream_t s) {
  if (n <= 0) {
    scan_empty<<<1, 1, 0, s>>>(out); MST_COUNT_LAUNCH();
    MST_CUDA_TRY(cudaGetLastError());
    return MST_OK;
  }
  const int64_t tiles = (n + SCAN_TILE - 1) / SCAN_TILE;
  scan_tile_sums<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(in, n, block_sums, enabled); MST_COUNT_LAUNCH();
  scan_sums_inplace<<<1, 1024, 0, s>>>(block_sums, tiles, enabled); MST_COUNT_LAUNCH();
  scan_tiles<<<(unsigned)tiles, SCAN_THREADS, 0, s>>>(in, n, block_sums, out, enabled); MST_COUNT_LAUNCH();
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}

mst_status_t mst_scan_i32(const int32_t* in, int32_t* out, int64_t n, int32_t* block_sums, cudaStream_t s) {
  return mst_scan_i32_if(in, out, n, block_sums, nullptr, s);
}

// bits[set] must be final.  Computes wscan[set], row_ptr[set], col_idx[set], vals[set].
mst_status_t mst_rebuild_from_bits(mst_layer* L, int set, const void* dense_W, int64_t ldw, int old_set,
                                   cudaStream_t s) {
  popc_words<<<blocks_for(L->nwords, 256), 256, 0, s>>>(L->bits[set], L->nwords, L->word_cnt); MST_COUNT_LAUNCH();
  MST_TRY(mst_scan_i32(L->word_cnt, L->wscan[set], L->nwords, L->block_sums, s));
  const unsigned grid = blocks_for(L->nwords * 32, 256);
  if (L->dtype == MST_F32) {
    fill_csr<float><<<grid, 256, 0, s>>>(L->bits[set], L->wscan[set], L->O, L->I, L->wpr, L->col_idx[set],
                                         (float*)L->vals[set], L->row_ptr[set], (const float*)dense_W, ldw,
                                         L->bits[old_set], L->wscan[old_set], (const float*)L->vals[old_set]); MST_COUNT_LAUNCH();
  } else {
    fill_csr<uint16_t><<<grid, 256, 0, s>>>(L->bits[set], L->wscan[set], L->O, L->I, L->wpr, L->col_idx[set],
                                            (uint16_t*)L->vals[set], L->row_ptr[set], (const uint16_t*)dense_W, ldw,
                                            L->bits[old_set], L->wscan[old_set], (const uint16_t*)L->vals[old_set]); MST_COUNT_LAUNCH();
  }
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}

// CSC view of the live set.
mst_status_t mst_build_csc(mst_layer* L, cudaStream_t s) {
  MST_TRY(mst_alloc_csc(L));
  const int c = L->cur;
  transpose_bits<<<blocks_for((int64_t)L->wpc * L->wpr * 32, 256), 256, 0, s>>>(L->bits[c], L->O, L->I, L->wpr, L->wpc,
                                                                                L->bitsT); MST_COUNT_LAUNCH();
  popc_words<<<blocks_for(L->nwordsT, 256), 256, 0, s>>>(L->bitsT, L->nwordsT, L->word_cnt); MST_COUNT_LAUNCH();
  MST_TRY(mst_scan_i32(L->word_cnt, L->wscanT, L->nwordsT, L->block_sums, s));
  fill_csc<<<blocks_for(L->nwordsT * 32, 256), 256, 0, s>>>(L->bitsT, L->wscanT, L->O, L->I, L->wpr, L->wpc, L->bits[c],
                                                            L->wscan[c], L->row_idx, L->perm, L->col_ptr); MST_COUNT_LAUNCH();
  MST_CUDA_TRY(cudaGetLastError());
  L->csc_valid = 1;
  return MST_OK;
}

mst_status_t mst_ensure_csc(const mst_layer* L, cudaStream_t s) {
  if (L->csc_valid) return MST_OK;
  return mst_build_csc(const_cast<mst_layer*>(L), s);
}

// new mask of an update from the three selection results; leaves popcounts in word_cnt
mst_status_t mst_combine_update_bits(mst_layer* L, int new_set, cudaStream_t s) {
  combine_bits<<<blocks_for(L->nwords, 256), 256, 0, s>>>(L->bits[L->cur], L->pruned_bits, L->grad_bits, L->rand_bits,
                                                          L->nwords, L->bits[new_set], L->word_cnt); MST_COUNT_LAUNCH();
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}

namespace {

// A pinned word that a kernel can write and the host reads after the synchronisation that mst_pack makes anyway: one per host
// thread, given back when the thread ends.
struct PinnedWord {
  int32_t* p = nullptr;
  int32_t* get() {
    if (!p && cudaHostAlloc((void**)&p, sizeof(int32_t), cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) p = nullptr;
    return p;
  }
  ~PinnedWord() {
    if (p) cudaFreeHost(p);
  }
};
thread_local PinnedWord t_pack_total;

// Blocks from which their counts are scanned by launches of their own: each block adding up what lies before it saves those launches,
// but its reads grow with the square of the blocks.  bf16, d = 0.05, added up / scanned: 26 / 36 us at 1120 blocks, 87 / 90 at 8192,
// 164 / 149 at 16384, 792 / 498 at 65536, 6650 / 1892 at 262140.
constexpr unsigned PACK_SCAN_BLOCKS = 10240;

// counts, scan: room for a word per block and one more (scan may be NULL below PACK_SCAN_BLOCKS); partials: for the scan
template <typename V, typename COL>
mst_status_t launch_pack(const uint8_t* mask, int O, int I, int wpr, const void* W, int64_t ldw, int64_t cap, uint32_t* bits, int32_t* counts,
                         int32_t* scan, int32_t* partials, int32_t* wscan, int32_t* row_ptr, COL* col_idx, void* vals, int32_t* total, cudaStream_t s) {
  const unsigned blocks = blocks_for((int64_t)O * wpr, PACK_WORDS);
  const int vec = (I % 32 == 0 && (reinterpret_cast<uintptr_t>(mask) & 15u) == 0) ? 1 : 0;
  MST_CUDA_TRY(mst_launch_overlapped(pack_bits_kernel, dim3(blocks), dim3(PACK_THREADS), 0, s, mask, O, I, wpr, vec, bits, counts));
  const int scanned = scan && blocks >= PACK_SCAN_BLOCKS ? 1 : 0;
  if (scanned) MST_TRY(mst_scan_i32(counts, scan, blocks, partials, s));
  MST_CUDA_TRY(mst_launch_overlapped(pack_fill_kernel<V, COL>, dim3(blocks), dim3(PACK_THREADS), 0, s, (const uint32_t*)bits,
                                     (const int32_t*)(scanned ? scan : counts), scanned, O, wpr, (const V*)W, ldw, cap, wscan, row_ptr, col_idx, (V*)vals,
                                     (volatile int32_t*)total));
  return MST_OK;
}

template <typename V>
mst_status_t launch_export(const int32_t* ptr, int n_ptr, const uint16_t* idx, const void* vals, int64_t nnz, int32_t* ptr_out,
                           int32_t* idx_out, void* vals_out, cudaStream_t s) {
  const int vec = ((reinterpret_cast<uintptr_t>(idx_out) | reinterpret_cast<uintptr_t>(vals_out)) & 15u) == 0 ? 1 : 0;
  const int64_t work = nnz / 4 + 1 > n_ptr ? nnz / 4 + 1 : n_ptr;
  const int64_t most = 16 * (int64_t)mst_sm_count(), blocks = (work + 255) / 256;
  MST_CUDA_TRY(mst_launch_overlapped(export_kernel<V>, dim3((unsigned)(blocks < most ? blocks : most)), dim3(256), 0, s, ptr, n_ptr, idx,
                                     (const V*)vals, nnz, ptr_out, idx_out, (V*)vals_out, vec));
  return MST_OK;
}

}  // namespace

extern "C" mst_status_t mst_pack(mst_layer_t* L, const void* W_dense, int64_t ldw, const uint8_t* mask,
                                 mst_stream_t stream) {
  if (!L || !W_dense || !mask) return MST_ERR_INVALID_ARG;
  if (ldw < L->I) return MST_ERR_SHAPE;
  cudaStream_t s = (cudaStream_t)stream;
  const int set = L->cur;
  L->nnz = -1;
  int32_t* total = t_pack_total.get();
  if (!total) return MST_ERR_CUDA;
  if (L->dtype == MST_F32)
    MST_TRY((launch_pack<float, uint16_t>(mask, L->O, L->I, L->wpr, W_dense, ldw, L->cap, L->bits[set], L->word_cnt, L->word_scan,
                                          L->block_sums, L->wscan[set], L->row_ptr[set], L->col_idx[set], L->vals[set], total, s)));
  else
    MST_TRY((launch_pack<uint16_t, uint16_t>(mask, L->O, L->I, L->wpr, W_dense, ldw, L->cap, L->bits[set], L->word_cnt, L->word_scan,
                                             L->block_sums, L->wscan[set], L->row_ptr[set], L->col_idx[set], L->vals[set], total, s)));
  MST_CUDA_TRY(cudaStreamSynchronize(s));
  const int32_t n = *(volatile int32_t*)total;
  if (n > L->cap) return MST_ERR_CAPACITY;
  L->nnz = n;
  ++L->version;
  // the CSC view serves the CUDA-core input gradient, the CSC export and the structure check: other layers get it on demand
  L->csc_valid = 0;
  if (mst_use_csc(L)) {
    MST_TRY(mst_build_csc(L, s));
    MST_CUDA_TRY(cudaStreamSynchronize(s));
  }
  return MST_OK;
}

extern "C" mst_status_t mst_export_csr(const mst_layer_t* L, int32_t* row_ptr, int32_t* col_idx, void* vals,
                                       mst_stream_t stream) {
  if (!L) return MST_ERR_INVALID_ARG;
  if (L->nnz < 0) return MST_ERR_NOT_PACKED;
  if (!row_ptr && !col_idx && !vals) return MST_OK;
  const int c = L->cur;
  return L->dtype == MST_F32 ? launch_export<float>(L->row_ptr[c], L->O + 1, L->col_idx[c], L->vals[c], L->nnz, row_ptr, col_idx, vals, (cudaStream_t)stream)
                             : launch_export<uint16_t>(L->row_ptr[c], L->O + 1, L->col_idx[c], L->vals[c], L->nnz, row_ptr, col_idx, vals, (cudaStream_t)stream);
}

extern "C" mst_status_t mst_export_csc(const mst_layer_t* L, int32_t* col_ptr, int32_t* row_idx, int32_t* perm,
                                       mst_stream_t stream) {
  if (!L) return MST_ERR_INVALID_ARG;
  if (L->nnz < 0) return MST_ERR_NOT_PACKED;
  cudaStream_t s = (cudaStream_t)stream;
  MST_TRY(mst_ensure_csc(L, s));
  if (!col_ptr && !row_idx && !perm) return MST_OK;
  return launch_export<float>(L->col_ptr, L->I + 1, L->row_idx, L->perm, L->nnz, col_ptr, row_idx, perm, s);   // 32-bit positions
}

extern "C" mst_status_t mst_validate(const mst_layer_t* L, mst_stream_t stream) {
  if (!L) return MST_ERR_INVALID_ARG;
  if (L->nnz < 0) return MST_ERR_NOT_PACKED;
  cudaStream_t s = (cudaStream_t)stream;
  const int c = L->cur;
  MST_TRY(mst_ensure_csc(L, s));
  validate_rows<<<blocks_for(L->O, 128), 128, 0, s>>>(L->row_ptr[c], L->col_idx[c], L->bits[c], L->O, L->I, L->wpr,
                                                     L->nnz, L->flags); MST_COUNT_LAUNCH();
  validate_cols<<<blocks_for(L->I, 128), 128, 0, s>>>(L->col_ptr, L->row_idx, L->perm, L->row_ptr[c], L->col_idx[c],
                                                     L->O, L->I, L->nnz, L->flags); MST_COUNT_LAUNCH();
  MST_CUDA_TRY(cudaGetLastError());
  int32_t f = 0;
  MST_CUDA_TRY(cudaMemcpyAsync(&f, L->flags, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  MST_CUDA_TRY(cudaStreamSynchronize(s));
  if (f) MST_CUDA_TRY(cudaMemsetAsync(L->flags, 0, sizeof(int32_t), s));  // reported once, then cleared
  if (f & MST_FLAG_CORRUPT) return MST_ERR_CORRUPT;
  if (f & MST_FLAG_NONFINITE) return MST_ERR_NONFINITE;
  return MST_OK;
}

// ---- allocation-free mask -> CSR ------------------------------------------------------------------------------------
// The same two launches as mst_pack, but with no handle and no allocation: the mask words and the blocks' entry counts live in one
// file-scope device array that every GPU loading this library holds until the process exits.
namespace {

constexpr int64_t NOALLOC_MAX_NUMEL = (int64_t)1 << 22;  // 4 194 304 entries, e.g. a 4096 x 1024 layer
constexpr int64_t NOALLOC_MAX_WORDS = (int64_t)1 << 18;  // >= numel/32 + rows for every shape accepted below
constexpr int64_t NOALLOC_SUMS = NOALLOC_MAX_WORDS / PACK_WORDS + 2;
static_assert(NOALLOC_MAX_WORDS / PACK_WORDS < PACK_SCAN_BLOCKS, "the counts are added up without a scan");
constexpr size_t NOALLOC_OFF_BITS = 0;
constexpr size_t NOALLOC_OFF_SUMS = NOALLOC_OFF_BITS + 4 * (size_t)NOALLOC_MAX_WORDS;
constexpr size_t NOALLOC_BYTES = NOALLOC_OFF_SUMS + 4 * (size_t)(NOALLOC_SUMS + 62);

static __device__ __align__(256) unsigned char g_noalloc_scratch[NOALLOC_BYTES];

constexpr int NOALLOC_MAX_DEVICES = 64;
unsigned char* g_noalloc_ptr[NOALLOC_MAX_DEVICES] = {};

// Device address of the scratch array on the current device.  g_noalloc_scratch itself is only a host-side handle
// for the symbol: the address a kernel can use has to be asked for, once per device, with that device current.
mst_status_t noalloc_scratch(unsigned char** out) {
  int devi = -1;
  MST_CUDA_TRY(cudaGetDevice(&devi));
  if (devi < 0 || devi >= NOALLOC_MAX_DEVICES) return MST_ERR_INVALID_ARG;
  if (!g_noalloc_ptr[devi]) {
    void* p = nullptr;
    MST_CUDA_TRY(cudaGetSymbolAddress(&p, g_noalloc_scratch));
    if (!p) return MST_ERR_CUDA;
    g_noalloc_ptr[devi] = (unsigned char*)p;
  }
  *out = g_noalloc_ptr[devi];
  return MST_OK;
}

}  // namespace

extern "C" mst_status_t mst_mask_to_csr_noalloc(int32_t O, int32_t I, mst_dtype_t dtype, const void* W_dense,
                                                int64_t ldw, const uint8_t* mask, int64_t nnz_capacity,
                                                int32_t* row_ptr, int32_t* col_idx, void* vals, mst_stream_t stream) {
  if (!W_dense || !mask || !row_ptr || !col_idx || !vals || nnz_capacity < 0) return MST_ERR_INVALID_ARG;
  if (dtype != MST_F32 && dtype != MST_BF16) return MST_ERR_DTYPE;
  if (O < 1 || I < 1 || O > 65535 || I > 65535 || ldw < I) return MST_ERR_SHAPE;
  const int wpr = (I + 31) / 32;
  const int64_t nwords = (int64_t)O * wpr;
  if ((int64_t)O * I > NOALLOC_MAX_NUMEL || nwords > NOALLOC_MAX_WORDS) return MST_ERR_CAPACITY;
  unsigned char* base = nullptr;
  MST_TRY(noalloc_scratch(&base));
  uint32_t* bits = (uint32_t*)(base + NOALLOC_OFF_BITS);
  int32_t* sums = (int32_t*)(base + NOALLOC_OFF_SUMS);
  cudaStream_t s = (cudaStream_t)stream;
  // every word of the scratch that the second launch reads is written by the first: nothing needs clearing
  if (dtype == MST_F32)
    return launch_pack<float, int32_t>(mask, O, I, wpr, W_dense, ldw, nnz_capacity, bits, sums, nullptr, nullptr, nullptr, row_ptr, col_idx, vals, nullptr, s);
  return launch_pack<uint16_t, int32_t>(mask, O, I, wpr, W_dense, ldw, nnz_capacity, bits, sums, nullptr, nullptr, nullptr, row_ptr, col_idx, vals, nullptr, s);
}
