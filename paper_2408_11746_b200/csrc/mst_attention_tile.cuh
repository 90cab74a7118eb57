// Pieces shared by the strided-attention kernels (Sec. 3.3): 64-row tiles as the TMA unit writes them, tcgen05 products of
// 128 x 64 score blocks with one operand in tensor memory, and the warp-level products that serve the far strided positions.
//
// Geometry: a tile holds 64 rows (tokens) of one head, 128 bytes a row, with the 128-byte swizzle (16-byte piece p of row r
// sits at piece p ^ (r & 7)); a block's own 128 rows are two such tiles one after the other.  Sequences and strides are
// multiples of 64, so a 64-row tile never mixes two sequences: whatever another sequence holds (inf and NaN too) stays out
// of the products, and a tile is either walked or left out.
#pragma once
#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdint>

#include "mst_internal.cuh"
#include "mst_tc_gemm.cuh"
#include "mst_tc_ptx.cuh"

namespace mst_att {

using namespace mst_ptx;

constexpr int D = 64;                      // head dimension
constexpr int ROWS = 128;                  // a block's own rows = tensor-memory lanes
constexpr int TS = 64;                     // rows of a streamed tile
constexpr int TILE_BYTES = TS * D * 2;     // 8 KiB
constexpr int LDF = 68;                    // row pitch of staged fp32 accumulators (floats)
constexpr int LDO = 72;                    // row pitch of staged bf16 results (elements)
constexpr float SCALE = 0.125f;            // 1 / sqrt(64)
constexpr float LOG2E = 1.4426950408889634f;
constexpr float SCALE_LOG2E = SCALE * LOG2E;   // exp(s / sqrt(d) - lse) = 2^(s * SCALE_LOG2E - lse * log2(e))

__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint64_t ex2_2(uint64_t v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return pack2(ex2(lo), ex2(hi));
}
__device__ __forceinline__ uint32_t pack_bf16_2(uint64_t v) {
  float lo, hi;
  unpack2(v, lo, hi);
  return pack_bf16(lo, hi);
}
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xFFFF0000u); }
// 16-byte piece of a swizzled tile (rows 128 bytes apart, also across neighbouring tiles)
__device__ __forceinline__ uint32_t piece_addr(uint32_t tile, int row, int piece) {
  return tile + (uint32_t)row * 128u + (((uint32_t)piece ^ (uint32_t)(row & 7)) << 4);
}
__device__ __forceinline__ uint4 lds128(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void prefetch_map(const CUtensorMap* tm) { asm volatile("prefetch.tensormap [%0];" ::"l"(tm) : "memory"); }
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst), "l"(src), "r"(bytes),
               "r"(bar)
               : "memory");
}
// the block's compute warps only (the producer and issuer lanes never join)
template <int THREADS>
__device__ __forceinline__ void compute_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(THREADS) : "memory");
}

// ---------------------------------------------------------------------------------------------- tcgen05 products
// instruction descriptor: fp32 accumulate, bf16 x bf16, M = 128, N = 64; b_mn: B stored with N contiguous
constexpr uint32_t IDESC_K = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(TS >> 3) << 17) | ((uint32_t)(ROWS >> 4) << 24);
constexpr uint32_t IDESC_MN = IDESC_K | (1u << 16);
// D[128 x 64] (+)= A (tensor memory, 128 rows x 16 bf16 in eight columns) * B (shared-memory descriptor)
__device__ __forceinline__ void tc_mma_ts(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
// scores: D = own rows (two tiles, K-major) * streamed tile^T over the 64 head dimensions
__device__ __forceinline__ void mma_scores(uint32_t tmem_d, uint64_t own, uint64_t tile) {
#pragma unroll
  for (int ks = 0; ks < D / 16; ++ks) tc_mma(tmem_d, own + (uint64_t)(ks * 2), tile + (uint64_t)(ks * 2), IDESC_K, ks > 0 ? 1u : 0u);
}
// D (+)= weights (tensor memory: those of 16 of the tile's rows in eight columns, `apart` columns from the next 16) * streamed tile
__device__ __forceinline__ void mma_weights(uint32_t tmem_d, uint32_t tmem_a, uint32_t apart, uint64_t tile, uint32_t accum) {
#pragma unroll
  for (int ks = 0; ks < TS / 16; ++ks)
    tc_mma_ts(tmem_d, tmem_a + (uint32_t)ks * apart, tile + (uint64_t)(ks * ((16 * 128) >> 4)), IDESC_MN, ks > 0 ? 1u : accum);
}
// sixteen fp32 columns of this warp's 32 lanes, and sixteen or eight packed ones back
__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_ld16_wait(uint32_t (&r)[16]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]), "+r"(r[8]), "+r"(r[9]),
                 "+r"(r[10]), "+r"(r[11]), "+r"(r[12]), "+r"(r[13]), "+r"(r[14]), "+r"(r[15])
               :
               : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%16], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15};" ::"r"(r[0]),
      "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]),
      "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%8], {%0, %1, %2, %3, %4, %5, %6, %7};" ::"r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// ---------------------------------------------------------------------------------------------- the tiles a block walks
// Own rows r0 .. r0 + 127 of a sequence.  LOOK_BACK: queries looking at keys; otherwise keys looking at the queries that see
// them.  First the `near` tiles (every pair at distance 0 .. l, so the first strided position too), then the far ones: tile
// (half, m) pairs the own rows r0 + 64 half + r with the rows m l away, row r with row r only, m >= 2.
// All quotients are of multiples of 64; `magic` = 2^32 / (l / 64) rounded up divides exactly while both sides are below 2^16 (0:
// plain division).  Four integer divisions were a tenth of a block's life.
__host__ __device__ inline uint32_t stride_magic(int l, int seq) {
  const uint32_t d = (uint32_t)l / TS;
  return (uint32_t)seq / TS < 65536u && d > 1 && d < 65536u ? (uint32_t)(((1ULL << 32) + d - 1) / d) : 0u;
}
__device__ __forceinline__ int strides_in(int n, int l, uint32_t magic) {
  return magic ? (int)__umulhi((uint32_t)n / TS, magic) : n / l;
}
template <bool LOOK_BACK>
struct Walk {
  int first, near, far0, far1, both, total;
  int r0, l;
  __device__ __forceinline__ Walk(int r0_, int l_, int seq, uint32_t magic) : r0(r0_), l(l_) {
    const bool second = r0 + TS < seq;       // the second half of the own rows lies inside the sequence
    int n0, n1;                              // strided positions of the halves, the first one included
    if (LOOK_BACK) {
      first = r0 - l > 0 ? r0 - l : 0;
      const int end = second ? r0 + ROWS : r0 + TS;
      near = (end - first) / TS;
      n0 = strides_in(r0, l, magic);
      n1 = strides_in(r0 + TS, l, magic);
    } else {
      first = r0;
      const int end = r0 + ROWS + l < seq ? r0 + ROWS + l : seq;
      near = (end - first) / TS;
      n0 = strides_in(seq - TS - r0, l, magic);
      n1 = second ? strides_in(seq - 2 * TS - r0, l, magic) : 0;
    }
    far0 = n0 > 1 ? n0 - 1 : 0;
    far1 = second && n1 > 1 ? n1 - 1 : 0;
    both = 2 * (far0 < far1 ? far0 : far1);
    total = near + far0 + far1;
  }
  // far tile f: which half of the own rows, and where the tile starts.  The halves take turns while both have tiles left, the one
  // with more of them first: the ring has an even number of stages, so each half keeps to stages of its own, sees every filling
  // of those and cannot take one for the next but one.
  __device__ __forceinline__ int far_half(int f) const {
    const int longer = far1 > far0 ? 1 : 0;
    return f < both ? (f & 1) ^ longer : longer;
  }
  // one half's far tiles: first, first + step, .. below far0 + far1
  __device__ __forceinline__ int far_step() const { return both > 0 ? 2 : 1; }
  __device__ __forceinline__ int far_first(int half) const {
    const int longer = far1 > far0 ? 1 : 0;
    return both > 0 ? half ^ longer : half == longer ? 0 : far0 + far1;
  }
  __device__ __forceinline__ int far_start(int f) const {
    const int m = f < both ? (f >> 1) + 2 : (both >> 1) + (f - both) + 2;
    const int own = r0 + TS * far_half(f);
    return LOOK_BACK ? own - m * l : own + m * l;
  }
  __device__ __forceinline__ int start(int j) const { return j < near ? first + j * TS : far_start(j - near); }
};

// The lane that feeds the ring.  A stage is given back by the commit behind the products of a near tile, or by the four warps that
// a far tile concerns (a barrier of its own: those warps cannot come to it again before the stage has been filled again).
template <int STAGES, typename W, typename Load, typename Wait>
__device__ __forceinline__ void feed_ring(const W& walk, uint32_t ring, uint32_t full, uint32_t empty, uint32_t far_done, Load load, Wait wait) {
  static_assert(STAGES % 2 == 0, "the halves' far tiles take turns");
  int s = 0;
  uint32_t lap = 0;
  for (int j = 0; j < walk.total; ++j) {
    const int before = j - STAGES;   // what the stage held one lap ago
    if (before >= 0) {
      const bool far = before >= walk.near;
      const uint32_t use = far ? (uint32_t)((before - walk.near) / STAGES) : lap - 1;
      if (!wait((far ? far_done : empty) + 8 * s, use & 1u)) return;
    }
    load(s, walk.start(j), ring + (uint32_t)(s * 2 * TILE_BYTES), full + 8 * s);
    if (++s == STAGES) { s = 0; ++lap; }
  }
}

// ---------------------------------------------------------------------------------------------- warp-level products (far tiles)
// mma.sync m16n8k16 with the published fragment layouts: with g = lane / 4 and t = lane % 4, an accumulator tile (16 x 8) holds
// rows g, g + 8 and columns 2t, 2t + 1; two neighbouring accumulator tiles, rounded to bf16, are the A operand of the next one.
__device__ __forceinline__ void ldsm_x4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
// rows r0 .. r0 + 15 of `own` times rows c0 .. c0 + 15 of `tile`, transposed: two 16 x 8 score tiles
__device__ __forceinline__ void far_scores(float (&c)[2][4], uint32_t own, int r0, uint32_t tile, int c0, int lane) {
#pragma unroll
  for (int nb = 0; nb < 2; ++nb) c[nb][0] = c[nb][1] = c[nb][2] = c[nb][3] = 0.f;
#pragma unroll
  for (int k2 = 0; k2 < 2; ++k2) {
    uint32_t b[2][4];
#pragma unroll
    for (int nb = 0; nb < 2; ++nb) ldsm_x4(b[nb], piece_addr(tile, c0 + nb * 8 + (lane & 7), k2 * 4 + (lane >> 3)));
#pragma unroll
    for (int kk = 0; kk < 2; ++kk) {
      uint32_t a[4];
      ldsm_x4(a, piece_addr(own, r0 + (lane & 7) + ((lane >> 3) & 1) * 8, (2 * k2 + kk) * 2 + (lane >> 4)));
#pragma unroll
      for (int nb = 0; nb < 2; ++nb) mma_bf16(c[nb], a, b[nb][2 * kk], b[nb][2 * kk + 1]);
    }
  }
}
// acc[16 x 16 N2] += weights (two 16 x 8 score tiles) * columns d0 .. of rows c0 .. c0 + 15 of `tile`
template <int N2>
__device__ __forceinline__ void far_accumulate(float (&acc)[2 * N2][4], const float (&w)[2][4], uint32_t tile, int c0, int d0, int lane) {
  const uint32_t a[4] = {pack_bf16(w[0][0], w[0][1]), pack_bf16(w[0][2], w[0][3]), pack_bf16(w[1][0], w[1][1]), pack_bf16(w[1][2], w[1][3])};
#pragma unroll
  for (int n2 = 0; n2 < N2; ++n2) {
    uint32_t b[4];
    ldsm_x4_t(b, piece_addr(tile, c0 + (lane & 7) + ((lane >> 3) & 1) * 8, d0 / 8 + n2 * 2 + (lane >> 4)));
    mma_bf16(acc[2 * n2], a, b[0], b[1]);
    mma_bf16(acc[2 * n2 + 1], a, b[2], b[3]);
  }
}
// This warp has read its rows of a far tile: its stage may be filled again.  The reads went through the generic proxy and the next
// copy into the stage goes through the async proxy, which an arrival alone does not order: without the proxy fence a read that was
// still under way now and then saw rows of the tile that came next (dQ at l = 128 differed from run to run in one of three calls;
// up to three tiles per half, as at l = 256, no stage is filled twice).  8 x 1024 tokens, 16 heads, l = 128: forward 35.2 -> 35.5 us,
// backward 107.8 -> 108.7.
__device__ __forceinline__ void far_release(uint32_t far_done, int lane) {
  fence_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive(far_done);
}
// this strip's accumulators -> fp32 rows r0 .. r0 + 15, columns d0 .., in shared memory (pitch LDF)
template <int NB>
__device__ __forceinline__ void far_stage(float* out, const float (&acc)[NB][4], int r0, int d0, int lane) {
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int nb = 0; nb < NB; ++nb) {
    *reinterpret_cast<float2*>(out + (r0 + g) * LDF + d0 + nb * 8 + 2 * t) = make_float2(acc[nb][0], acc[nb][1]);
    *reinterpret_cast<float2*>(out + (r0 + g + 8) * LDF + d0 + nb * 8 + 2 * t) = make_float2(acc[nb][2], acc[nb][3]);
  }
}

// ---------------------------------------------------------------------------------------------- results
// sixteen columns of one row: the accumulator, the far tiles' share of it if there is one, scaled, as bf16 into the staged
// result tile (pitch LDO)
__device__ __forceinline__ void stage_row(__nv_bfloat16* out, int row, int col, const uint32_t (&v)[16], const float* sums, float scale) {
  float x[16];
#pragma unroll
  for (int e = 0; e < 16; ++e) x[e] = __uint_as_float(v[e]);
  if (sums) {
#pragma unroll
    for (int e = 0; e < 16; e += 4) {
      const float4 y = *reinterpret_cast<const float4*>(sums + row * LDF + col + e);
      x[e] += y.x; x[e + 1] += y.y; x[e + 2] += y.z; x[e + 3] += y.w;
    }
  }
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    uint4 w;
    w.x = pack_bf16(x[8 * g + 0] * scale, x[8 * g + 1] * scale);
    w.y = pack_bf16(x[8 * g + 2] * scale, x[8 * g + 3] * scale);
    w.z = pack_bf16(x[8 * g + 4] * scale, x[8 * g + 5] * scale);
    w.w = pack_bf16(x[8 * g + 6] * scale, x[8 * g + 7] * scale);
    *reinterpret_cast<uint4*>(out + row * LDO + col + 8 * g) = w;
  }
}
// rows first .. first + N - 1 of the staged tile -> global rows, eight lanes per row of 128 bytes
template <int N>
__device__ __forceinline__ void write_rows(const __nv_bfloat16* staged, int first, __nv_bfloat16* out, int64_t row, int64_t ld, int lane) {
#pragma unroll
  for (int it = 0; it < N / 4; ++it) {
    const int r = first + it * 4 + (lane >> 3), piece = lane & 7;
    *reinterpret_cast<uint4*>(out + (row + r) * ld + piece * 8) = *reinterpret_cast<const uint4*>(staged + r * LDO + piece * 8);
  }
}

// [rows x cols] bf16, ld elements between rows; box = 64 rows x 64 columns (one head of 64 tokens)
inline bool tile_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)D, (cuuint32_t)TS};
  cuuint32_t estr[2] = {1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace mst_att
