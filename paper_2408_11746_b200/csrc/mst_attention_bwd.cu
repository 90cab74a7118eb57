// Strided sparse self-attention, backward (Sec. 3.3): gradients of
//   Out[i] = sum_{j in S_i} P_ij v_j,   P = softmax over S_i of q_i . k_j / sqrt(d),
//   S_i = { j <= i : i - j < l  or  (i - j) mod l == 0 }
// with respect to q, k and v, from the upstream gradient dOut, the forward output and its stored log-sum-exp:
//   delta_i = dOut_i . Out_i                     (= sum_j P_ij dP_ij)
//   P_ij    = exp(q_i . k_j / sqrt(d) - lse_i)   dP_ij = dOut_i . v_j      dS_ij = P_ij (dP_ij - delta_i)
//   dV_j = sum_i P_ij dOut_i      dK_j = sum_i dS_ij q_i / sqrt(d)      dQ_i = sum_j dS_ij k_j / sqrt(d)
//
// Two launches, no atomics (every output element has one owner and a fixed summation order):
//   1. dQ, query-centric: a block owns 128 queries of one (sequence, head) and walks 64-key tiles.  It forms delta first and
//      leaves (-lse log2 e, delta) of its rows in the scratch buffer for the second launch.
//   2. dK and dV, key-centric: a block owns 128 keys and walks the 64-query tiles that see them, on the transposed scores.
// Roles of a block's ten warps:
//   warps 0-7  algebra: thread = own row (tensor-memory lane), the two warps of a lane quarter take 32 of a tile's 64 columns each.
//              Scores and dP come from tensor memory, dS (and P) go back as bf16 and are the A operand of the second products
//              where they lie, so nothing score-shaped passes through shared memory;
//   warp 8     one lane feeds a four-tile ring by TMA;
//   warp 9     one lane issues tcgen05.mma: S = Q K^T, dP = dOut V^T (128 x 64), then dQ += dS K, or dV += P^T dOut, dK += dS^T Q.
// 256 columns of tensor memory and 102 KiB of shared memory: two blocks per SM, so that one block's products run while
// the other's algebra does.  The far strided positions (i - 2l, i - 3l, ...: one key per query and distance) are visited
// after the window as tiles of which only the diagonal counts: warp-level mma.sync products of 16 rows each, whose sums are
// added to the accumulators when the rows leave.
// Measured at 16 x 1024 tokens, 12 heads: l = 256 144 us, l = 128 (8 x 1024, 16 heads) 109 us; the two mma.sync kernels and the delta
// kernel before took 219 and 117 us.  Of 148 and 112 us, leaving out the far tiles gives 124 and 75 us, the window's tiles beyond the first as well 67
// and 47 us (300 and 200 MB of compulsory traffic in two passes: 46 and 31 us); the exponentials cost 2 us.
#include <cuda.h>
#include <cuda_bf16.h>

#include "mst_attention_tile.cuh"
#include "mst_internal.cuh"

namespace {
using namespace mst_att;

constexpr int CW = 8;                              // algebra warps (16 x 1024 tokens, 12 heads, l = 256, the call: 4 - 165 us, 8 - 148, 16 - 171)
constexpr int PARTS = CW / 4;                      // warps of a lane quarter: they share a tile's 64 columns
constexpr int COLS = TS / PARTS;                   // columns of one warp ...
constexpr int PIECES = COLS / 16;                  // ... in pieces of sixteen
constexpr int STRIPS = ROWS / 16 / CW;             // 16-row strips of a warp in the far tiles' products
constexpr int THREADS = 32 * (CW + 2);
constexpr int STAGES = 4;
constexpr int STAT_BYTES = TS * 8;                 // -lse log2 e of a tile's queries, then their -delta
constexpr int RING_BYTES = STAGES * 2 * TILE_BYTES;
constexpr int TMEM_COLS = 256;

__device__ int g_bwd_error = 0;

struct BwdParams {
  const __nv_bfloat16* Out;
  int64_t ldo;
  const float* lse;    // [batch, heads, seq]
  float* stat;         // [batch, heads, seq / 64][2][64]: -lse log2 e, -delta
  __nv_bfloat16 *dQ, *dK, *dV;
  int64_t ldg;
  int seq, heads, stride;
  uint32_t magic;
};

// shared memory of a block, 1024-byte aligned: the own rows of two operands, the ring, the ring's statistics, barriers
struct Smem {
  uint32_t own0, own1, ring, stat, full, empty, own_full, s_full, s_free, w_full, w_free, acc_full, dp_full, p_full, far_done;
  unsigned char* base;
  __device__ __forceinline__ explicit Smem(unsigned char* raw) {
    const uint32_t a = (smem_u32(raw) + 1023u) & ~1023u;
    base = raw + (a - smem_u32(raw));
    own0 = a;
    own1 = own0 + 2 * TILE_BYTES;
    ring = own1 + 2 * TILE_BYTES;
    stat = ring + RING_BYTES;
    full = stat + STAGES * STAT_BYTES + PARTS * ROWS * 4 + ROWS * 8;
    empty = full + 8 * STAGES;
    own_full = empty + 8 * STAGES;
    s_full = own_full + 8;
    s_free = s_full + 8;
    w_full = s_free + 8;
    w_free = w_full + 8;
    acc_full = w_free + 8;
    dp_full = acc_full + 8;
    p_full = dp_full + 8;
    far_done = p_full + 8;
  }
  template <typename T>
  __device__ __forceinline__ T* at(uint32_t addr) const {
    return reinterpret_cast<T*>(base + (addr - own0));
  }
};
constexpr size_t SMEM_BYTES = 4 * TILE_BYTES + RING_BYTES + STAGES * STAT_BYTES + PARTS * ROWS * 4 + ROWS * 8 + 24 * STAGES + 80 + 1024;
static_assert(ROWS * LDF * 4 <= RING_BYTES, "staged sums must fit the ring");
static_assert(ROWS * LDO * 2 <= 4 * TILE_BYTES, "staged results must fit the own tiles");

__device__ __forceinline__ bool wait_on(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait(bar, parity, abort_flag, &g_bwd_error);
}

__device__ __forceinline__ uint32_t block_setup(const Smem& S, uint32_t* holder, int* abort_sh, int warp) {
  if (threadIdx.x == 0) {
    *abort_sh = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(S.full + 8 * s, 1);
      mbar_init(S.empty + 8 * s, 1);
      mbar_init(S.far_done + 8 * s, CW / 2);
    }
    mbar_init(S.own_full, 1);
    mbar_init(S.s_full, 1);
    mbar_init(S.dp_full, 1);
    mbar_init(S.s_free, CW);
    mbar_init(S.w_full, CW);
    mbar_init(S.p_full, CW);
    mbar_init(S.w_free, 1);
    mbar_init(S.acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == CW + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(holder)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  return *holder;
}
__device__ __forceinline__ void block_teardown(uint32_t tmem, int warp, volatile int* abort_flag) {
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);   // let copies and products in flight land
  }
  tc_fence_before();
  __syncthreads();
  if (warp == CW + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

// The lane that feeds the ring: the block's own rows of two operands, then tile after tile of two others (and, for the
// keys' pass, the statistics of the tile's queries).
template <typename W>
__device__ __forceinline__ void feed(const Smem& S, const W& walk, const CUtensorMap* own_a, const CUtensorMap* own_b,
                                     const CUtensorMap* tile_a, const CUtensorMap* tile_b, int col, int row0, const float* stat,
                                     volatile int* abort_flag) {
  mbar_expect_tx(S.own_full, 4 * TILE_BYTES);
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    tma_load_2d(S.own0 + t * TILE_BYTES, own_a, col, row0 + walk.r0 + t * TS, S.own_full);
    tma_load_2d(S.own1 + t * TILE_BYTES, own_b, col, row0 + walk.r0 + t * TS, S.own_full);
  }
  feed_ring<STAGES>(walk, S.ring, S.full, S.empty, S.far_done, [&](int s, int at, uint32_t dst, uint32_t bar) {
    mbar_expect_tx(bar, 2 * TILE_BYTES + (stat ? STAT_BYTES : 0));
    tma_load_2d(dst, tile_a, col, row0 + at, bar);
    tma_load_2d(dst + TILE_BYTES, tile_b, col, row0 + at, bar);
    if (stat) bulk_load(S.stat + s * STAT_BYTES, stat + 2 * at, STAT_BYTES, bar);
  }, [&](uint32_t bar, uint32_t parity) { return wait_on(bar, parity, abort_flag); });
}

// ------------------------------------------------------------------------------------------- dQ
// Tensor memory: S in columns 0-63, dP 64-127, dQ 128-191, dS (bf16) 192-223.  S and dP are free as soon as they are in
// registers, so the next tile's scores are formed during this tile's algebra.
__global__ void __launch_bounds__(THREADS, 2)
attn_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const BwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const Smem S(smem_raw);
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, b = blockIdx.z, q0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * ROWS, l = P.stride;
  const int row0 = b * P.seq;
  const Walk<true> walk(q0, l, P.seq, P.magic);
  if (warp == CW && lane < 4) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : &tmG);
  const uint32_t tmem = block_setup(S, &holder, &abort_sh, warp);
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  if (warp == CW) {
    if (lane == 0) feed(S, walk, &tmQ, &tmG, &tmK, &tmV, h * D, row0, nullptr, abort_flag);
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t qd = smem_desc(S.own0, 16, 1024), gd = smem_desc(S.own1, 16, 1024), kd0 = smem_desc(S.ring, 16, 1024);
      const uint64_t step = (2 * TILE_BYTES) >> 4, vofs = TILE_BYTES >> 4;
      bool ok = wait_on(S.own_full, 0, abort_flag);
      int s = 0, sp = 0;
      uint32_t ph = 0;
      for (int j = 0; j <= walk.near && ok; ++j) {
        if (j < walk.near) {
          ok = wait_on(S.full + 8 * s, ph, abort_flag) && (j == 0 || wait_on(S.s_free, (uint32_t)(j - 1) & 1u, abort_flag));
          if (!ok) break;
          tc_fence_after();
          mma_scores(tmem, qd, kd0 + step * (uint32_t)s);
          mma_scores(tmem + 64, gd, kd0 + step * (uint32_t)s + vofs);
          tc_commit(S.s_full);
        }
        if (j > 0) {
          ok = wait_on(S.w_full, (uint32_t)(j - 1) & 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          mma_weights(tmem + 128, tmem + 192, 8, kd0 + step * (uint32_t)sp, j > 1 ? 1u : 0u);
          tc_commit(S.empty + 8 * sp);
          tc_commit(j == walk.near ? S.acc_full : S.w_free);
        }
        sp = s;
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
  } else {
    const int quarter = warp & 3, c = (warp >> 2) * COLS;    // this warp's lanes, and its share of a tile's 64 columns
    const int r = quarter * 32 + lane, i = q0 + r;
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
    float* part = S.at<float>(S.stat + STAGES * STAT_BYTES);                  // [PARTS][128] partial sums of delta
    float2* stat_s = reinterpret_cast<float2*>(part + PARTS * ROWS);              // the rows' -lse log2 e and delta
    // delta of this row: the threads of a row take COLS dimensions each
    const bool row_ok = i < P.seq;
    const int64_t st = ((int64_t)b * P.heads + h) * P.seq + i;
    uint4 o[COLS / 8];
    float nl = 0.f;
    if (row_ok) {
      const uint4* src = reinterpret_cast<const uint4*>(P.Out + ((int64_t)row0 + i) * P.ldo + h * D + c);
#pragma unroll
      for (int p = 0; p < COLS / 8; ++p) o[p] = __ldg(src + p);
      nl = -__ldg(P.lse + st) * LOG2E;
    }
    bool ok = wait_on(S.own_full, 0, abort_flag);
    float del = 0.f;
    if (row_ok) {
#pragma unroll
      for (int p = 0; p < COLS / 8; ++p) {
        const uint4 g = lds128(piece_addr(S.own1, r, c / 8 + p));
        const uint32_t ow[4] = {o[p].x, o[p].y, o[p].z, o[p].w}, gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          del = fmaf(bf_lo(ow[e]), bf_lo(gw[e]), del);
          del = fmaf(bf_hi(ow[e]), bf_hi(gw[e]), del);
        }
      }
    }
    part[c / COLS * ROWS + r] = del;
    compute_sync<32 * CW>();
    del = 0.f;
#pragma unroll
    for (int p = 0; p < PARTS; ++p) del += part[p * ROWS + r];
    if (c == 0) {
      stat_s[r] = make_float2(nl, del);
      if (row_ok) {
        float* out = P.stat + (st / TS) * (2 * TS) + r % TS;   // st = r modulo 64
        out[0] = nl;
        out[TS] = -del;
      }
    }

    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E), nl2 = pack2(nl, nl), ndel2 = pack2(-del, -del);
    const int i_lo = q0 + quarter * 32;                      // this warp's rows: i_lo .. i_lo + 31
    for (int j = 0; j < walk.near && ok; ++j) {
      ok = wait_on(S.s_full, (uint32_t)j & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t s[PIECES][16], dp[PIECES][16], w[PIECES][8];
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        tmem_ld16_nowait(t_row + (uint32_t)(c + pc * 16), s[pc]);
        tmem_ld16_nowait(t_row + (uint32_t)(64 + c + pc * 16), dp[pc]);
      }
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        tmem_ld16_wait(s[pc]);
        tmem_ld16_wait(dp[pc]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(S.s_free);
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        const int k0 = walk.first + j * TS + c + pc * 16;    // the piece's keys: k0 .. k0 + 15
        if (i_lo + 31 >= k0 && i_lo - (k0 + 15) <= l) {      // some pair is attended
#pragma unroll
          for (int e = 0; e < 8; ++e) {
            const uint64_t pp = ex2_2(fma2(pack2(s[pc][2 * e], s[pc][2 * e + 1]), scale2, nl2));
            w[pc][e] = pack_bf16_2(mul2(pp, add2(pack2(dp[pc][2 * e], dp[pc][2 * e + 1]), ndel2)));
          }
          if (!(i_lo >= k0 + 15 && i_lo + 31 - k0 <= l)) {   // some pair is not
            const int back0 = i - k0;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              if ((unsigned)(back0 - 2 * e) > (unsigned)l) w[pc][e] &= 0xFFFF0000u;
              if ((unsigned)(back0 - 2 * e - 1) > (unsigned)l) w[pc][e] &= 0x0000FFFFu;
            }
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) w[pc][e] = 0u;
        }
      }
      if (j > 0) {
        ok = wait_on(S.w_free, (uint32_t)(j - 1) & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
      }
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) tmem_st8(t_row + (uint32_t)(192 + c / 2 + pc * 8), w[pc]);
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(S.w_full);
    }

    // far tiles: warp = STRIPS times 16 rows of the block, with the keys in line with them
    const int far = walk.far0 + walk.far1;
    const int r0 = warp * 16 * STRIPS;
    float acc[STRIPS][8][4];
#pragma unroll
    for (int sp = 0; sp < STRIPS; ++sp)
#pragma unroll
      for (int nb = 0; nb < 8; ++nb) acc[sp][nb][0] = acc[sp][nb][1] = acc[sp][nb][2] = acc[sp][nb][3] = 0.f;
    if (far > 0) {
      compute_sync<32 * CW>();                               // the rows' statistics are in place
      const int g = lane >> 2, t = lane & 3;
      const int step = walk.far_step();
      for (int place = walk.near + walk.far_first(r0 >> 6); place < walk.total; place += step) {
        const int s = place % STAGES;
        ok = wait_on(S.full + 8 * s, (uint32_t)(place / STAGES) & 1u, abort_flag);
        if (!ok) break;
        const uint32_t kt = S.ring + s * 2 * TILE_BYTES;
#pragma unroll
        for (int sp = 0; sp < STRIPS; ++sp) {
          const int rs = r0 + sp * 16, c0 = rs & 63;
          const float2 st0 = stat_s[rs + g], st1 = stat_s[rs + g + 8];
          float sc[2][4], dp[2][4];
          far_scores(sc, S.own0, rs, kt, c0, lane);
          far_scores(dp, S.own1, rs, kt + TILE_BYTES, c0, lane);
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float ds = 0.f;
              if (g + (e >> 1) * 8 == nb * 8 + 2 * t + (e & 1)) {
                const float p = ex2(fmaf(sc[nb][e], SCALE_LOG2E, (e >> 1) ? st1.x : st0.x));
                ds = p * (dp[nb][e] - ((e >> 1) ? st1.y : st0.y));
              }
              sc[nb][e] = ds;
            }
          }
          far_accumulate<4>(acc[sp], sc, kt, c0, 0, lane);
        }
        far_release(S.far_done + 8 * s, lane);
      }
    }
    ok = ok && wait_on(S.acc_full, 0, abort_flag);
    tc_fence_after();
    // every product has completed and every tile has been consumed: the ring takes the far sums, the own tiles the results
    uint32_t v[PIECES][16];
#pragma unroll
    for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(128 + c + pc * 16), v[pc]);
    compute_sync<32 * CW>();
    float* sums = far > 0 ? S.at<float>(S.ring) : nullptr;
    __nv_bfloat16* res = S.at<__nv_bfloat16>(S.own0);
    if (far > 0) {
#pragma unroll
      for (int sp = 0; sp < STRIPS; ++sp) far_stage<8>(sums, acc[sp], r0 + sp * 16, 0, lane);
      compute_sync<32 * CW>();
    }
#pragma unroll
    for (int pc = 0; pc < PIECES; ++pc) {
      tmem_ld16_wait(v[pc]);
      stage_row(res, r, c + pc * 16, v[pc], sums, SCALE);
    }
    compute_sync<32 * CW>();
    constexpr int N = ROWS / CW;   // rows a warp writes
    if (ok && q0 + warp * N < P.seq) write_rows<N>(res, warp * N, P.dQ + h * D, (int64_t)row0 + q0, P.ldg, lane);
  }
  block_teardown(tmem, warp, abort_flag);
}

// ------------------------------------------------------------------------------------------- dK, dV
// Tensor memory: S^T in columns 0-63, dP^T 64-127, dK 128-191, dV 192-255; each warp writes P^T over the scores it has
// read (eight columns at its sixteen's start) and dS^T over its dP.
__global__ void __launch_bounds__(THREADS, 2)
attn_bwd_dkv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const BwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const Smem S(smem_raw);
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, b = blockIdx.z, k0 = (int)blockIdx.x * ROWS, l = P.stride;   // early keys have the most tiles
  const int row0 = b * P.seq;
  const Walk<false> walk(k0, l, P.seq, P.magic);
  if (warp == CW && lane < 4) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : &tmG);
  const uint32_t tmem = block_setup(S, &holder, &abort_sh, warp);
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  if (warp == CW) {
    if (lane == 0)
      feed(S, walk, &tmK, &tmV, &tmQ, &tmG, h * D, row0, P.stat + 2 * ((int64_t)b * P.heads + h) * P.seq, abort_flag);
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t kd = smem_desc(S.own0, 16, 1024), vd = smem_desc(S.own1, 16, 1024), qd0 = smem_desc(S.ring, 16, 1024);
      const uint64_t step = (2 * TILE_BYTES) >> 4, gofs = TILE_BYTES >> 4;
      bool ok = wait_on(S.own_full, 0, abort_flag);
      int s = 0;
      uint32_t ph = 0;
      for (int j = 0; j < walk.near && ok; ++j) {
        ok = wait_on(S.full + 8 * s, ph, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint64_t qd = qd0 + step * (uint32_t)s;
        // Everything executes in issue order, so the scores may overwrite the P of the tile before (its dV product is issued)
        // and dP its dS.  S goes ahead of the last tile's dK: the exponentials start while dK and dP are formed.
        if (j == 0) mma_scores(tmem, kd, qd);
        if (j == 0) tc_commit(S.s_full);
        mma_scores(tmem + 64, vd, qd + gofs);
        tc_commit(S.dp_full);
        ok = wait_on(S.p_full, (uint32_t)j & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
        mma_weights(tmem + 192, tmem, 16, qd + gofs, j > 0 ? 1u : 0u);
        if (j + 1 < walk.near) {
          const int sn = s + 1 == STAGES ? 0 : s + 1;
          ok = wait_on(S.full + 8 * sn, sn ? ph : ph ^ 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          mma_scores(tmem, kd, qd0 + step * (uint32_t)sn);
          tc_commit(S.s_full);
        }
        ok = wait_on(S.w_full, (uint32_t)j & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
        mma_weights(tmem + 128, tmem + 64, 16, qd, j > 0 ? 1u : 0u);
        tc_commit(S.empty + 8 * s);
        if (j + 1 == walk.near) tc_commit(S.acc_full);
        if (++s == STAGES) { s = 0; ph ^= 1u; }
      }
    }
  } else {
    const int quarter = warp & 3, c = (warp >> 2) * COLS;    // this warp's lanes, and its share of a tile's 64 columns
    const int r = quarter * 32 + lane, jk = k0 + r;
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E);
    const int j_lo = k0 + quarter * 32;                      // this warp's keys: j_lo .. j_lo + 31
    bool ok = wait_on(S.own_full, 0, abort_flag);
    int s = 0;
    uint32_t ph = 0;
    for (int j = 0; j < walk.near && ok; ++j) {
      const uint32_t sa = S.stat + (uint32_t)(s * STAT_BYTES + c * 4);
      ok = wait_on(S.full + 8 * s, ph, abort_flag) &&        // the statistics have landed too
           wait_on(S.s_full, (uint32_t)j & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
      uint32_t w[PIECES][8], st[PIECES][16];
      uint64_t p[PIECES][8];                                 // P^T of this row, fp32 pairs
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(c + pc * 16), st[pc]);
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        const int q0 = walk.first + j * TS + c + pc * 16;    // the piece's queries: q0 .. q0 + 15
        tmem_ld16_wait(st[pc]);
        if (q0 + 15 >= j_lo && q0 - (j_lo + 31) <= l) {      // some pair is attended
#pragma unroll
          for (int e = 0; e < 4; ++e) {                      // statistics of four queries at a time
            const uint4 nl = lds128(sa + 64u * pc + 16u * e);
            p[pc][2 * e] = ex2_2(fma2(pack2(st[pc][4 * e], st[pc][4 * e + 1]), scale2, pack2(nl.x, nl.y)));
            p[pc][2 * e + 1] = ex2_2(fma2(pack2(st[pc][4 * e + 2], st[pc][4 * e + 3]), scale2, pack2(nl.z, nl.w)));
          }
          if (!(q0 >= j_lo + 31 && q0 + 15 - j_lo <= l)) {   // some pair is not
            const int back0 = q0 - jk;
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              float lo, hi;
              unpack2(p[pc][e], lo, hi);
              p[pc][e] = pack2((unsigned)(back0 + 2 * e) > (unsigned)l ? 0.f : lo, (unsigned)(back0 + 2 * e + 1) > (unsigned)l ? 0.f : hi);
            }
          }
        } else {
#pragma unroll
          for (int e = 0; e < 8; ++e) p[pc][e] = 0ULL;
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) w[pc][e] = pack_bf16_2(p[pc][e]);
        tmem_st8(t_row + (uint32_t)(c + pc * 16), w[pc]);
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(S.p_full);
      ok = wait_on(S.dp_full, (uint32_t)j & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(64 + c + pc * 16), st[pc]);
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        const int q0 = walk.first + j * TS + c + pc * 16;
        tmem_ld16_wait(st[pc]);
        if (q0 + 15 >= j_lo && q0 - (j_lo + 31) <= l) {
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const uint4 nd = lds128(sa + (uint32_t)(TS * 4) + 64u * pc + 16u * e);
            w[pc][2 * e] = pack_bf16_2(mul2(p[pc][2 * e], add2(pack2(st[pc][4 * e], st[pc][4 * e + 1]), pack2(nd.x, nd.y))));
            w[pc][2 * e + 1] = pack_bf16_2(mul2(p[pc][2 * e + 1], add2(pack2(st[pc][4 * e + 2], st[pc][4 * e + 3]), pack2(nd.z, nd.w))));
          }
          if (!(q0 >= j_lo + 31 && q0 + 15 - j_lo <= l)) {
            const int back0 = q0 - jk;
#pragma unroll
            for (int e = 0; e < 8; ++e)
              w[pc][e] &= ((unsigned)(back0 + 2 * e) > (unsigned)l ? 0u : 0x0000FFFFu) |
                          ((unsigned)(back0 + 2 * e + 1) > (unsigned)l ? 0u : 0xFFFF0000u);
          }
        }
        tmem_st8(t_row + (uint32_t)(64 + c + pc * 16), w[pc]);   // zeros where nothing is attended
      }
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(S.w_full);
      if (++s == STAGES) { s = 0; ph ^= 1u; }
    }

    // far tiles: warp = STRIPS times 16 keys of the block, with the queries in line with them
    const int far = walk.far0 + walk.far1;
    const int r0 = warp * 16 * STRIPS;
    float acc_k[STRIPS][8][4], acc_v[STRIPS][8][4];
#pragma unroll
    for (int sp = 0; sp < STRIPS; ++sp)
#pragma unroll
      for (int nb = 0; nb < 8; ++nb) {
        acc_k[sp][nb][0] = acc_k[sp][nb][1] = acc_k[sp][nb][2] = acc_k[sp][nb][3] = 0.f;
        acc_v[sp][nb][0] = acc_v[sp][nb][1] = acc_v[sp][nb][2] = acc_v[sp][nb][3] = 0.f;
      }
    if (far > 0) {
      const int g = lane >> 2, t = lane & 3;
      const int step = walk.far_step();
      for (int place = walk.near + walk.far_first(r0 >> 6); place < walk.total; place += step) {
        const int s = place % STAGES;
        ok = wait_on(S.full + 8 * s, (uint32_t)(place / STAGES) & 1u, abort_flag);
        if (!ok) break;
        const uint32_t qt = S.ring + s * 2 * TILE_BYTES;
#pragma unroll
        for (int sp = 0; sp < STRIPS; ++sp) {
          const int rs = r0 + sp * 16, c0 = rs & 63;
          float st[2][4], dp[2][4];
          far_scores(st, S.own0, rs, qt, c0, lane);
          far_scores(dp, S.own1, rs, qt + TILE_BYTES, c0, lane);
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
            const float* sq = S.at<float>(S.stat + (uint32_t)(s * STAT_BYTES)) + c0 + nb * 8 + 2 * t;
            const float2 nl = *reinterpret_cast<const float2*>(sq), nd = *reinterpret_cast<const float2*>(sq + TS);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float p = 0.f, ds = 0.f;
              if (g + (e >> 1) * 8 == nb * 8 + 2 * t + (e & 1)) {
                p = ex2(fmaf(st[nb][e], SCALE_LOG2E, (e & 1) ? nl.y : nl.x));
                ds = p * (dp[nb][e] + ((e & 1) ? nd.y : nd.x));
              }
              st[nb][e] = p;
              dp[nb][e] = ds;
            }
          }
          far_accumulate<4>(acc_v[sp], st, qt + TILE_BYTES, c0, 0, lane);
          far_accumulate<4>(acc_k[sp], dp, qt, c0, 0, lane);
        }
        far_release(S.far_done + 8 * s, lane);
      }
    }
    ok = ok && wait_on(S.acc_full, 0, abort_flag);
    tc_fence_after();
    compute_sync<32 * CW>();   // every product has completed and every tile has been consumed
    float* sums = far > 0 ? S.at<float>(S.ring) : nullptr;
    __nv_bfloat16* res = S.at<__nv_bfloat16>(S.own0);
    constexpr int N = ROWS / CW;   // rows a warp writes
#pragma unroll
    for (int which = 0; which < 2; ++which) {   // dK, then dV
      uint32_t v[PIECES][16];
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(128 + which * 64 + c + pc * 16), v[pc]);
      if (far > 0) {
#pragma unroll
        for (int sp = 0; sp < STRIPS; ++sp) far_stage<8>(sums, which ? acc_v[sp] : acc_k[sp], r0 + sp * 16, 0, lane);
      }
      if (far > 0 || which) compute_sync<32 * CW>();   // the sums are in place, dK's rows have left the staging tile
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        tmem_ld16_wait(v[pc]);
        stage_row(res, r, c + pc * 16, v[pc], sums, which ? 1.f : SCALE);
      }
      compute_sync<32 * CW>();
      if (ok && k0 + warp * N < P.seq) write_rows<N>(res, warp * N, (which ? P.dV : P.dK) + h * D, (int64_t)row0 + k0, P.ldg, lane);
    }
  }
  block_teardown(tmem, warp, abort_flag);
}

}  // namespace

mst_status_t mst_attention_bwd_error_flags(int32_t* flags) {
  int v = 0;
  MST_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_bwd_error, sizeof(int)));
  *flags = v;
  return MST_OK;
}

extern "C" mst_status_t mst_strided_attention_bwd(const void* Q, const void* K, const void* V, int64_t ld, const void* Out,
                                                  int64_t ldo, const void* dOut, int64_t lddo, const float* lse,
                                                  int32_t batch, int32_t seq_len, int32_t heads, int32_t head_dim,
                                                  int32_t stride, void* dQ, void* dK, void* dV, int64_t ldg,
                                                  mst_stream_t stream) {
  if (!Q || !K || !V || !Out || !dOut || !lse || !dQ || !dK || !dV || batch < 0 || seq_len <= 0 || heads <= 0)
    return MST_ERR_INVALID_ARG;
  if (head_dim != D || seq_len % TS != 0 || stride <= 0 || stride % TS != 0) return MST_ERR_SHAPE;
  const int64_t width = (int64_t)heads * D;
  if (ld < width || ldo < width || lddo < width || ldg < width || ld % 8 || ldo % 8 || lddo % 8 || ldg % 8) return MST_ERR_SHAPE;
  if (((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V) |
        reinterpret_cast<uintptr_t>(Out) | reinterpret_cast<uintptr_t>(dOut) | reinterpret_cast<uintptr_t>(dQ) |
        reinterpret_cast<uintptr_t>(dK) | reinterpret_cast<uintptr_t>(dV)) & 15u) != 0)
    return MST_ERR_SHAPE;
  if (batch == 0) return MST_OK;
  const int64_t rows = (int64_t)batch * seq_len;
  if (rows > 0x7FFFFFFF || heads > 65535 || batch > 65535) return MST_ERR_SHAPE;
  cudaStream_t s = (cudaStream_t)stream;
  CUtensorMap tmQ, tmK, tmV, tmG;
  if (!tile_map(&tmQ, Q, rows, width, ld) || !tile_map(&tmK, K, rows, width, ld) || !tile_map(&tmV, V, rows, width, ld) ||
      !tile_map(&tmG, dOut, rows, width, lddo))
    return MST_ERR_SHAPE;
  void* ws = nullptr;
  MST_TRY(mst_workspace_kind(MST_WS_ATTENTION, 2 * sizeof(float) * (size_t)rows * heads, &ws));
  BwdParams P;
  P.Out = (const __nv_bfloat16*)Out;
  P.ldo = ldo;
  P.lse = lse; P.stat = (float*)ws;
  P.dQ = (__nv_bfloat16*)dQ; P.dK = (__nv_bfloat16*)dK; P.dV = (__nv_bfloat16*)dV;
  P.ldg = ldg;
  P.seq = seq_len; P.heads = heads;
  P.stride = stride < seq_len ? stride : seq_len;   // from there on the same pairs: all earlier positions
  P.magic = stride_magic(P.stride, seq_len);
  MST_SMEM_LIMIT((attn_bwd_dq_kernel), SMEM_BYTES);
  MST_SMEM_LIMIT((attn_bwd_dkv_kernel), SMEM_BYTES);
  dim3 grid((unsigned)((seq_len + ROWS - 1) / ROWS), (unsigned)heads, (unsigned)batch);
  MST_CUDA_TRY(mst_launch_overlapped(attn_bwd_dq_kernel, grid, dim3(THREADS), SMEM_BYTES, s, tmQ, tmK, tmV, tmG, P));
  MST_CUDA_TRY(mst_launch_overlapped(attn_bwd_dkv_kernel, grid, dim3(THREADS), SMEM_BYTES, s, tmQ, tmK, tmV, tmG, P));
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}
