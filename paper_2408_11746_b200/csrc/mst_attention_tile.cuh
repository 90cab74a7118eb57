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

#include <cmath>
#include <cstdint>
#include <numeric>

#include "mst_internal.cuh"
#include "mst_tc_gemm.cuh"
#include "mst_tc_ptx.cuh"

namespace mst_att {

using namespace mst_ptx;

constexpr int D = 64;                      // head dimension
constexpr int ROWS = 128;                  // a block's own rows = tensor-memory lanes
constexpr int TS = 64;                     // rows of a streamed tile
constexpr int TILE_BYTES = TS * D * 2;     // 8 KiB
constexpr int SLOT_BYTES = 2 * TILE_BYTES; // a ring slot: a tile of each of two operands, or 128 rows of results on their way out
constexpr int CW = 8;                      // algebra warps: thread = row, the two warps of a lane quarter share a tile's columns
constexpr int THREADS = 32 * (CW + 2);     // and the lane that loads, the lane that issues the products
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
__device__ __forceinline__ void mbar_arrive_n(uint32_t bar, uint32_t n) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(n) : "memory");
}

// ---------------------------------------------------------------------------------------------- one block after another
// A block that runs takes over blocks of its own grid that have not started (cluster launch control), so that the next one's
// operands are on their way while this one's last products and results are.  The request goes out at a block's start, its answer (16 bytes
// by the async proxy) is read by every role at the block's end; a proxy fence of the reader's, before it lets go of the next block's own
// rows, orders that ahead of the answer after next, which comes to the same place.  No request follows one that found nothing left.
// The block to come is claimed when its predecessor starts, not by whoever is done first, so it pays where each of those that run at once has more
// than two to see to (MORE): at 297 of 296 blocks 9 x 384 tokens, 11 heads, l = 128 took 40.0 us with it, 33.9 without, 3 x 1536, 9 heads, l = 192 (324) 63.7
// and 50.0, 5 x 1152, 13 heads, l = 256 (585) 75.1 and 71.9, 3 x 2048, 14 heads, l = 128 (672) 114.0 and 118.2, 6 x 1024, 17 heads, l = 256 (816) 97.3
// and 101.1.
// Fewer blocks leave all of this out: its instructions alone cost a launch 0.4 us.  Their results
// leave as whole rows by the warps, which nothing follows: through a ring slot and the TMA unit they took 0.3 us a kernel longer.  What a block
// walks is worked out ahead of the wait for the kernel before, and windows that reach back half of the sequence or more, so that
// there are no far tiles, have kernels without them (FAR: 0.4 us a kernel for code that is only jumped over, as the kernels of a pass take turns in the
// instruction cache).  Forward and backward, before / after each of these: 1 x 256 tokens, 6 heads, l = 256 23.3 / 21.8 / 22.0 / 21.6 us,
// 2 x 512, 12 heads, l = 256 33.8 / 33.0 / 32.2 / 31.9, 3 x 768, 15 heads, l = 512 49.6 / 49.6 / 49.3 / 48.6; with far tiles 3 x 640, 9 heads, l = 128
// 38.3 / 37.3 / 37.1.  (Rows stored straight from the registers, 16 bytes of each at a time: 1 to 3 us longer.)
// Grid: heads, batch, blocks of a sequence, those with the most tiles first.  (Blocks fastest, as their keys and values are then found in
// L2, left the SMs idle for a quarter of the time at the end: 8 x 1024 tokens, 16 heads, l = 128 have 3.5 blocks for each of the
// 296 that run at once; 16 x 1024 tokens, 12 heads, l = 256 backward 153.6 -> 132.6 us by the order.)  Where four operands exceed L2
// it is gone through in equal parts that do not, as few as possible, of the batch or of the heads or of both, or far tiles and the
// next kernel's rows come from DRAM (9 x 1792 tokens, 20 heads, forward and backward 338 -> 321 us in three parts, 16 x 2048, 20 heads, l = 128 922 -> 737;
// 16 x 1024, 12 heads, which fit: 169 in one part, 174 in two, 177 in four.  Each part starts with its heaviest blocks again, so many small parts cost as
// well: 13 x 1024 tokens, 20 heads, l = 128 246 us in thirteen parts of the batch, 229 in two of the heads; 13 x 1664, 13 heads, l = 512, where thirteen is
// the least, 348 in them and 339 in one, with a seventh more than L2 holds.)
// Grids that run at once (two blocks to an SM, no last wave to fill) have a sequence's blocks first where the window is shorter than the sequence, so that blocks with
// tiles in common are neighbours: forward and backward 1 x 1024 tokens, 6 heads, l = 128 43.3 -> 39.6 us, 2 x 1024, 9 heads, l = 256 42.5 -> 40.2; windows
// of the whole sequence lose by it (3 x 512, 10 heads 39.3 -> 41.9, 2 x 256, 20 heads 26.8 -> 28.4).
// Sequences of more blocks than the grid's third dimension holds have them in its first.
struct Place { int h, b, block; };
constexpr int GRID_Z = 65535;
constexpr double L2_BYTES = 126e6;
__device__ __forceinline__ Place place(int x, int y, int z, int blocks, int heads, bool blocks_first) {
  if (blocks_first || blocks > GRID_Z) return Place{y, z, x};
  while (z >= blocks) {   // the next part
    z -= blocks;
    x += (int)gridDim.x;
    if (x >= heads) {
      x -= heads;
      y += (int)gridDim.y;
    }
  }
  return Place{x, y, z};
}
inline dim3 place_grid(int heads, int batch, int blocks, bool blocks_first) {
  if (blocks_first || blocks > GRID_Z) return dim3((unsigned)blocks, (unsigned)heads, (unsigned)batch);
  const double share = 4.0 * 2.0 * (double)blocks * ROWS * heads * D * batch / L2_BYTES;
  int of_batch = 1, of_heads = 1;
  const int64_t least = (int64_t)ceil(share);
  for (int64_t parts = least; least > 1 && parts <= 8 * least; ++parts) {
    const int64_t g = std::gcd(parts, (int64_t)batch);
    if (heads % (parts / g) == 0) {
      of_batch = (int)g;
      of_heads = (int)(parts / g);
      break;
    }
  }
  if ((int64_t)blocks * of_batch * of_heads > GRID_Z || (share < 1.3 && of_batch * of_heads > 4)) of_batch = of_heads = 1;
  return dim3((unsigned)(heads / of_heads), (unsigned)(batch / of_batch), (unsigned)(blocks * of_batch * of_heads));
}
struct Form { bool more, far, blocks_first; };
inline Form form_of(int batch, int heads, int blocks, int stride, int seq) {
  const int64_t all = (int64_t)batch * heads * blocks, at_once = 2 * (int64_t)mst_sm_count();
  return Form{all > 2 * at_once, seq - stride > stride, all <= at_once && stride < seq};
}
__device__ __forceinline__ void take_over(uint32_t answer, uint32_t bar) {
  mbar_expect_tx(bar, 16);
  asm volatile("clusterlaunchcontrol.try_cancel.async.shared::cta.mbarrier::complete_tx::bytes.b128 [%0], [%1];" ::"r"(answer), "r"(bar) : "memory");
}
__device__ __forceinline__ bool taken_over(uint32_t answer, Place& p, int blocks, int heads) {
  uint32_t ok, x, y, z;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b128 r;\n\t"
      "ld.shared.b128 r, [%4];\n\t"
      "clusterlaunchcontrol.query_cancel.is_canceled.pred.b128 p, r;\n\t"
      "selp.u32 %3, 1, 0, p;\n\t"
      "mov.u32 %0, 0;\n\tmov.u32 %1, 0;\n\tmov.u32 %2, 0;\n\t"
      "@p clusterlaunchcontrol.query_cancel.get_first_ctaid.v4.b32.b128 {%0, %1, %2, _}, r;\n\t}"
      : "=r"(x), "=r"(y), "=r"(z), "=r"(ok)
      : "r"(answer)
      : "memory");
  p = place((int)x, (int)y, (int)z, blocks, heads, false);
  return ok != 0;
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
// them.  First the far tiles: tile (half, m) pairs the own rows r0 + 64 half + r with the rows m l away, row r with row r only,
// m >= 2; their sums become the start of the tensor-memory accumulators.  Then the `near` tiles: every pair at distance 0 .. l, so
// the first strided position too.
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
  // worked out here, not where it is first used
  __device__ __forceinline__ void now() { asm volatile("" : "+r"(first), "+r"(near), "+r"(far0), "+r"(far1), "+r"(both), "+r"(total)); }
  // far tile f: which half of the own rows, and where the tile starts.  The halves take turns while both have tiles left, the one
  // with more of them first, and the ring has an even number of slots: each half's tiles come in slots of its own.
  __device__ __forceinline__ int far() const { return far0 + far1; }
  __device__ __forceinline__ int far_half(int f) const {
    const int longer = far1 > far0 ? 1 : 0;
    return f < both ? (f & 1) ^ longer : longer;
  }
  // one half's far tiles: far_first, far_first + far_step, .. below far()
  __device__ __forceinline__ int far_step() const { return both > 0 ? 2 : 1; }
  __device__ __forceinline__ int far_first(int half) const {
    const int longer = far1 > far0 ? 1 : 0;
    return both > 0 ? half ^ longer : half == longer ? 0 : far();
  }
  __device__ __forceinline__ int far_start(int f) const {
    const int m = f < both ? (f >> 1) + 2 : (both >> 1) + (f - both) + 2;
    const int own = r0 + TS * far_half(f);
    return LOOK_BACK ? own - m * l : own + m * l;
  }
  __device__ __forceinline__ int start(int j) const { return j < far() ? far_start(j) : first + (j - far()) * TS; }
};

// A running position in the ring.  Slots are used in one order: far tiles, near tiles, slots for the results, block after block.  A
// parity cannot tell a filling from the next but one, so nobody may wait for a slot whose last filling he cannot know to be over:
// the warps of a half meet their own far tiles only, in slots of their own; then everybody meets (far_over), and what is not waited
// for after that is known by the scores or by the results.  A slot is given back by eight arrivals: two from each of the four warps
// that a far tile concerns, seven of the issuing lane's and the commit behind a near tile's last product, one from each warp for results.
constexpr uint32_t SLOT_ARRIVALS = CW;
template <int STAGES>
struct Ring {
  static_assert(STAGES % 2 == 0, "the halves' far tiles take turns");
  uint32_t s = 0, lap = 0;
  __device__ __forceinline__ void next() {
    if (++s == STAGES) { s = 0; ++lap; }
  }
  __device__ __forceinline__ void skip(int n) {
    s += (uint32_t)n;
    lap += s / STAGES;
    s %= STAGES;
  }
};

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
// acc[16 x 64] += weights (two 16 x 8 score tiles) * rows c0 .. c0 + 15 of `tile`
__device__ __forceinline__ void far_accumulate(float (&acc)[8][4], const float (&w)[2][4], uint32_t tile, int c0, int lane) {
  const uint32_t a[4] = {pack_bf16(w[0][0], w[0][1]), pack_bf16(w[0][2], w[0][3]), pack_bf16(w[1][0], w[1][1]), pack_bf16(w[1][2], w[1][3])};
#pragma unroll
  for (int n2 = 0; n2 < 4; ++n2) {
    uint32_t b[4];
    ldsm_x4_t(b, piece_addr(tile, c0 + (lane & 7) + ((lane >> 3) & 1) * 8, n2 * 2 + (lane >> 4)));
    mma_bf16(acc[2 * n2], a, b[0], b[1]);
    mma_bf16(acc[2 * n2 + 1], a, b[2], b[3]);
  }
}
// sums of a warp-level product (16 rows x 64 columns, eight 16 x 8 accumulator tiles) -> sixteen lanes from taddr's on, 64 columns
__device__ __forceinline__ void tmem_st_tiles(uint32_t taddr, const float (&a)[8][4]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%32], "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};" ::"f"(a[0][0]),
      "f"(a[0][1]), "f"(a[0][2]), "f"(a[0][3]), "f"(a[1][0]), "f"(a[1][1]), "f"(a[1][2]), "f"(a[1][3]), "f"(a[2][0]), "f"(a[2][1]),
      "f"(a[2][2]), "f"(a[2][3]), "f"(a[3][0]), "f"(a[3][1]), "f"(a[3][2]), "f"(a[3][3]), "f"(a[4][0]), "f"(a[4][1]), "f"(a[4][2]),
      "f"(a[4][3]), "f"(a[5][0]), "f"(a[5][1]), "f"(a[5][2]), "f"(a[5][3]), "f"(a[6][0]), "f"(a[6][1]), "f"(a[6][2]), "f"(a[6][3]),
      "f"(a[7][0]), "f"(a[7][1]), "f"(a[7][2]), "f"(a[7][3]), "r"(taddr)
      : "memory");
}
// ---------------------------------------------------------------------------------------------- far tiles: two lanes a row
// Row r of the own rows meets row r % 64 of the tile and no other, so a far tile is 64 dot products and 64 scaled rows.  A warp takes
// sixteen rows, lanes i and i + 16 the two halves of row i's 64 columns: every byte is read from shared memory once.  fp32 sums of
// exact bf16 products (the mixed-precision FMA of sm_100); weights are rounded to bf16 like those of the near tiles. 8 x 1024 tokens,
// 16 heads, l = 128 forward: 28.4 us, and 30.6 with mma.sync products as in the backward kernels.
__device__ __forceinline__ void fma_bf16(float& acc, uint16_t a, uint16_t b) { asm("fma.rn.f32.bf16 %0, %1, %2, %0;" : "+f"(acc) : "h"(a), "h"(b)); }
__device__ __forceinline__ void halves(uint32_t w, uint16_t& lo, uint16_t& hi) { asm("mov.b32 {%0, %1}, %2;" : "=h"(lo), "=h"(hi) : "r"(w)); }
struct FarRow { uint32_t w[16]; };   // 32 columns
__device__ __forceinline__ FarRow far_row(uint32_t tile, int row, int lane) {
  FarRow x;
#pragma unroll
  for (int p = 0; p < 4; ++p) {
    const uint4 v = lds128(piece_addr(tile, row, (lane >> 4) * 4 + p));
    x.w[4 * p] = v.x; x.w[4 * p + 1] = v.y; x.w[4 * p + 2] = v.z; x.w[4 * p + 3] = v.w;
  }
  return x;
}
// the whole row's dot product, in both of its lanes
__device__ __forceinline__ float far_dot(const FarRow& a, const FarRow& b) {
  float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    uint16_t al, ah, bl, bh;
    halves(a.w[e], al, ah);
    halves(b.w[e], bl, bh);
    fma_bf16(s[e & 1], al, bl);
    fma_bf16(s[2 + (e & 1)], ah, bh);
  }
  const float x = (s[0] + s[1]) + (s[2] + s[3]);
  return x + __shfl_xor_sync(0xffffffffu, x, 16);
}
__device__ __forceinline__ void far_add(float (&acc)[32], float weight, const FarRow& b) {
  uint16_t w, dummy;
  halves(pack_bf16(weight, 0.f), w, dummy);
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    uint16_t lo, hi;
    halves(b.w[e], lo, hi);
    fma_bf16(acc[2 * e], w, lo);
    fma_bf16(acc[2 * e + 1], w, hi);
  }
}
// the sums -> sixteen tensor-memory lanes from taddr's on, 64 columns: the start of an accumulator
__device__ __forceinline__ void far_start_sums(uint32_t taddr, const float (&a)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x32bx2.x32.b32 [%32], 32, "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31};" ::"f"(a[0]),
      "f"(a[1]), "f"(a[2]), "f"(a[3]), "f"(a[4]), "f"(a[5]), "f"(a[6]), "f"(a[7]), "f"(a[8]), "f"(a[9]), "f"(a[10]), "f"(a[11]),
      "f"(a[12]), "f"(a[13]), "f"(a[14]), "f"(a[15]), "f"(a[16]), "f"(a[17]), "f"(a[18]), "f"(a[19]), "f"(a[20]), "f"(a[21]),
      "f"(a[22]), "f"(a[23]), "f"(a[24]), "f"(a[25]), "f"(a[26]), "f"(a[27]), "f"(a[28]), "f"(a[29]), "f"(a[30]), "f"(a[31]), "r"(taddr)
      : "memory");
}
// This warp has read its rows of a far tile: its stage may be filled again.  The reads went through the generic proxy and the next
// copy into the stage goes through the async proxy, which an arrival alone does not order: without the proxy fence a read that was
// still under way now and then saw rows of the tile that came next (dQ at l = 128 differed from run to run in one of three calls;
// up to three tiles per half, as at l = 256, no stage is filled twice).  8 x 1024 tokens, 16 heads, l = 128: forward 35.2 -> 35.5 us,
// backward 107.8 -> 108.7.
__device__ __forceinline__ void far_release(uint32_t empty, int lane) {
  fence_async_smem();
  __syncwarp();
  if (lane == 0) mbar_arrive_n(empty, SLOT_ARRIVALS / 4);
}

// ---------------------------------------------------------------------------------------------- results
// sixteen columns of one row, scaled, as bf16 into a slot that holds 128 result rows (swizzled like a tile)
__device__ __forceinline__ void stage_row(uint32_t slot, int row, int col, const uint32_t (&v)[16], float scale) {
#pragma unroll
  for (int g = 0; g < 2; ++g) {
    uint32_t w[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) w[e] = pack_bf16(__uint_as_float(v[8 * g + 2 * e]) * scale, __uint_as_float(v[8 * g + 2 * e + 1]) * scale);
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(piece_addr(slot, row, col / 8 + g)), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3])
                 : "memory");
  }
}
// sixteen rows of the slot from `first` on -> the caller's rows, eight lanes per row of 128 bytes
__device__ __forceinline__ void write_rows(uint32_t slot, int first, __nv_bfloat16* out, int64_t ld, int lane) {
#pragma unroll
  for (int it = 0; it < 4; ++it) {
    const int r = first + it * 4 + (lane >> 3);
    *reinterpret_cast<uint4*>(out + r * ld + (lane & 7) * 8) = lds128(piece_addr(slot, r, lane & 7));
  }
}
// [rows x cols] bf16, ld elements between rows; box = 64 rows x 64 columns (one head of 64 tokens), or the 32 rows of a lane quarter's results
inline bool tile_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows = TS) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)D, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace mst_att
