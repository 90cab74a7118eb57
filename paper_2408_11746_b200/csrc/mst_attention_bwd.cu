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
//      leaves (-lse log2 e, -delta) of its rows in the scratch buffer for the second launch.
//   2. dK and dV, key-centric: a block owns 128 keys and walks the 64-query tiles that see them, on the transposed scores.
// Roles of a block's ten warps:
//   warps 0-7  algebra: thread = own row (tensor-memory lane), the two warps of a lane quarter take 32 of a tile's 64 columns each.
//              Scores and dP come from tensor memory, dS (and P) go back as bf16 and are the A operand of the second products
//              where they lie, so nothing score-shaped passes through shared memory;
//   warp 8     one lane feeds a four-slot ring by TMA;
//   warp 9     one lane issues tcgen05.mma: S = Q K^T, dP = dOut V^T (128 x 64), then dQ += dS K, or dV += P^T dOut, dK += dS^T Q.
// 256 columns of tensor memory and 102 KiB of shared memory: two blocks per SM, so that one block's products run while
// the other's algebra does.  The far strided positions (i - 2l, i - 3l, ...: one key per query and distance) come first, as tiles
// of which only the diagonal counts: warp-level mma.sync products of 16 rows each, whose sums are where the tensor-memory accumulators
// start (formed row by row on the FMA pipe, as the forward kernel does it, they take a third more instructions here: 128.4 us against 126.6 at l = 256).
// A block that is done takes over one that has not started; its own rows, the forward output and the first tiles are then in
// shared memory or on their way.  Results leave by TMA from slots of the ring, or, in a block without
// successors, as whole rows from where the own rows were.
// Bound: as forward, the chain of a tile through its warps.
// 16 x 1024 tokens, 12 heads, l = 256 144.7 -> 124.2 us, 8 x 1024, 16 heads, l = 128 108.7 -> 87.8.
#include <cuda.h>
#include <cuda_bf16.h>

#include "mst_attention_tile.cuh"
#include "mst_internal.cuh"

namespace {
using namespace mst_att;

constexpr int PARTS = CW / 4;                      // warps of a lane quarter: they share a tile's 64 columns
constexpr int COLS = TS / PARTS;                   // columns of one warp ...
constexpr int PIECES = COLS / 16;                  // ... in pieces of sixteen
constexpr int STAGES = 4;
constexpr int STAT_BYTES = TS * 8;                 // -lse log2 e of a tile's queries, then their -delta
constexpr int TMEM_COLS = 256;

__device__ int g_bwd_error = 0;

struct BwdParams {
  const __nv_bfloat16* Out;
  int64_t ldo;
  const float* lse;    // [batch, heads, seq]
  float* stat;         // [batch, heads, seq / 64][2][64]: -lse log2 e, -delta
  __nv_bfloat16 *dQ, *dK, *dV;
  int64_t ldg;
  int seq, heads, stride, blocks, blocks_first;
  uint32_t magic;
};

// shared memory of a block, 1024-byte aligned: the own rows of two operands, the ring, the ring's statistics, partial sums of
// the rows' delta, answers, barriers
struct Smem {
  uint32_t own0, own1, ring, stat, part, answers, full, empty, own_full, own_free, s_full, s_free, w_full, w_free, acc_full, dp_full, p_full,
      next_full, pair0, far_over;
  unsigned char* base;
  __device__ __forceinline__ explicit Smem(unsigned char* raw) {
    const uint32_t a = (smem_u32(raw) + 1023u) & ~1023u;
    base = raw + (a - smem_u32(raw));
    own0 = a;
    own1 = own0 + 2 * TILE_BYTES;
    ring = own1 + 2 * TILE_BYTES;
    stat = ring + STAGES * SLOT_BYTES;
    part = stat + STAGES * STAT_BYTES;
    answers = part + PARTS * ROWS * 4;
    full = answers + 32;
    empty = full + 8 * STAGES;
    own_full = empty + 8 * STAGES;
    own_free = own_full + 8;
    s_full = own_free + 8;
    s_free = s_full + 8;
    w_full = s_free + 8;
    w_free = w_full + 8;
    acc_full = w_free + 8;
    dp_full = acc_full + 8;
    p_full = dp_full + 8;
    next_full = p_full + 8;
    pair0 = next_full + 16;
    far_over = pair0 + 32;
  }
  template <typename T>
  __device__ __forceinline__ T* at(uint32_t addr) const {
    return reinterpret_cast<T*>(base + (addr - own0));
  }
};
constexpr size_t SMEM_BYTES = 4 * TILE_BYTES + STAGES * SLOT_BYTES + STAGES * STAT_BYTES + PARTS * ROWS * 4 + 32 + 16 * STAGES + 16 * 8 + 1024;

__device__ __forceinline__ bool wait_on(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait(bar, parity, abort_flag, &g_bwd_error);
}

__device__ __forceinline__ uint32_t block_setup(const Smem& S, uint32_t* holder, int* abort_sh, int warp) {
  if (threadIdx.x == 0) {
    *abort_sh = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(S.full + 8 * s, 1);
      mbar_init(S.empty + 8 * s, SLOT_ARRIVALS);
    }
    mbar_init(S.own_full, 1);
    mbar_init(S.own_free, 1 + CW);
    mbar_init(S.s_full, 1);
    mbar_init(S.dp_full, 1);
    mbar_init(S.s_free, CW);
    mbar_init(S.w_full, CW);
    mbar_init(S.p_full, CW);
    mbar_init(S.w_free, 1);
    mbar_init(S.acc_full, 1);
    for (int e = 0; e < 2; ++e) mbar_init(S.next_full + 8 * e, 1);
    for (int e = 0; e < 4; ++e) mbar_init(S.pair0 + 8 * e, PARTS);
    mbar_init(S.far_over, CW);
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

// block `it` of this one's life is at its end: the next one, if there is one (the warps' fence comes with the own rows' release)
template <bool MORE>
__device__ __forceinline__ bool next_block(const Smem& S, const BwdParams& P, int it, Place& at, volatile int* abort_flag) {
  return MORE && wait_on(S.next_full + 8 * (it & 1), (uint32_t)(it >> 1) & 1u, abort_flag) && taken_over(S.answers + 16 * (it & 1), at, P.blocks, P.heads);
}
// the two warps of a lane quarter meet
__device__ __forceinline__ bool meet(const Smem& S, int quarter, uint32_t parity, int lane, volatile int* abort_flag) {
  __syncwarp();
  if (lane == 0) mbar_arrive(S.pair0 + 8 * quarter);
  return wait_on(S.pair0 + 8 * quarter, parity, abort_flag);
}

// The lane that loads: the block's own rows of two operands (and, for the queries' pass, their forward output, in a slot), then tile after tile of two others (and, for the keys' pass, the
// statistics of the tile's queries), then RESULTS slots that the results leave through.
template <bool LOOK_BACK, int RESULTS, bool MORE>
__device__ __forceinline__ void feed(const Smem& S, const BwdParams& P, Place at, const Walk<LOOK_BACK>& first, const CUtensorMap* own_a, const CUtensorMap* own_b,
                                     const CUtensorMap* tile_a, const CUtensorMap* tile_b, const CUtensorMap* own_out, volatile int* abort_flag) {
  Ring<STAGES> k;
  bool ok = true;
  auto slot = [&]() { return k.lap == 0 || wait_on(S.empty + 8 * k.s, (k.lap - 1) & 1u, abort_flag); };
  for (int it = 0; ok; ++it) {
    const int col = at.h * D, row0 = at.b * P.seq;
    const Walk<LOOK_BACK> walk = MORE ? Walk<LOOK_BACK>((LOOK_BACK ? P.blocks - 1 - at.block : at.block) * ROWS, P.stride, P.seq, P.magic) : first;
    const float* stat = LOOK_BACK ? nullptr : P.stat + 2 * ((int64_t)at.b * P.heads + at.h) * P.seq;
    if (it > 0 && !wait_on(S.own_free, (uint32_t)(it - 1) & 1u, abort_flag)) return;
    mbar_expect_tx(S.own_full, 4 * TILE_BYTES);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      tma_load_2d(S.own0 + t * TILE_BYTES, own_a, col, row0 + walk.r0 + t * TS, S.own_full);
      tma_load_2d(S.own1 + t * TILE_BYTES, own_b, col, row0 + walk.r0 + t * TS, S.own_full);
    }
    if (MORE) take_over(S.answers + 16 * (it & 1), S.next_full + 8 * (it & 1));
    if (LOOK_BACK && MORE) {
      if (!slot()) return;
      mbar_expect_tx(S.full + 8 * k.s, 2 * TILE_BYTES);
#pragma unroll
      for (int t = 0; t < 2; ++t) tma_load_2d(S.ring + k.s * SLOT_BYTES + t * TILE_BYTES, own_out, col, row0 + walk.r0 + t * TS, S.full + 8 * k.s);
      k.next();
    }
    for (int j = 0; j < walk.total; ++j) {
      if (!slot()) return;
      const int from = walk.start(j);
      const uint32_t dst = S.ring + k.s * SLOT_BYTES, bar = S.full + 8 * k.s;
      mbar_expect_tx(bar, 2 * TILE_BYTES + (LOOK_BACK ? 0 : STAT_BYTES));
      tma_load_2d(dst, tile_a, col, row0 + from, bar);
      tma_load_2d(dst + TILE_BYTES, tile_b, col, row0 + from, bar);
      if (!LOOK_BACK) bulk_load(S.stat + k.s * STAT_BYTES, stat + 2 * from, STAT_BYTES, bar);
      k.next();
    }
    if (!MORE) return;
    for (int e = 0; e < RESULTS; ++e) {
      if (!slot()) return;
      mbar_arrive(S.full + 8 * k.s);
      k.next();
    }
    ok = next_block<MORE>(S, P, it, at, abort_flag);
    fence_async_smem();
  }
}

// ------------------------------------------------------------------------------------------- dQ
// Tensor memory: S in columns 0-63, dP 64-127, dQ 128-191, dS (bf16) 192-223.  S and dP are free as soon as they are in
// registers, so the next tile's scores are formed during this tile's algebra.
template <bool MORE, bool FAR>   // see mst_attention_tile.cuh
__global__ void __launch_bounds__(THREADS, 2)
attn_bwd_dq_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                   const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmO,
                   const __grid_constant__ CUtensorMap tmD, const BwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const Smem S(smem_raw);
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = P.stride;
  if (warp == CW && lane < (MORE ? 6 : 4)) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : lane == 3 ? &tmG : lane == 4 ? &tmO : &tmD);
  const uint32_t tmem = block_setup(S, &holder, &abort_sh, warp);
  Place at = place((int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, P.blocks, P.heads, !MORE && P.blocks_first);
  Walk<true> first((P.blocks - 1 - at.block) * ROWS, l, P.seq, P.magic);
  if (!MORE) first.now();
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  if (warp == CW) {
    if (lane == 0) feed<true, 1, MORE>(S, P, at, first, &tmQ, &tmG, &tmK, &tmV, &tmO, abort_flag);
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t qd = smem_desc(S.own0, 16, 1024), gd = smem_desc(S.own1, 16, 1024), kd0 = smem_desc(S.ring, 16, 1024);
      const uint64_t step = SLOT_BYTES >> 4, vofs = TILE_BYTES >> 4;
      Ring<STAGES> k;
      uint32_t t = 0;   // near tiles so far
      bool ok = true;
      auto filled = [&]() { return wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag); };
      for (int it = 0; ok; ++it) {
        const Walk<true> walk = MORE ? Walk<true>((P.blocks - 1 - at.block) * ROWS, l, P.seq, P.magic) : first;
        const uint32_t from_far = FAR && walk.far() > 0 ? 1u : 0u;
        const int skip = (MORE ? 1 : 0) + walk.far();        // the forward output, the far tiles
        ok = wait_on(S.own_full, (uint32_t)it & 1u, abort_flag);
        // A slot's parity tells one filling from the next only if the one before is known to be over.  The slots skipped here are filled once the
        // far tiles are over; in a block without successors the first two tiles' scores go ahead of that, beside delta and the far tiles, where
        // their slots are filled for the first time.  Everything later waits for weights of all warps, and these come after the far
        // tiles' sums.  3 x 512 tokens, 10 heads, l = 512, forward and backward 40.6 -> 39.5 us, 3 x 640, 9 heads, l = 128 unchanged; in blocks
        // with successors it gains nothing (8 x 1024, 16 heads, l = 128: 0.6 % lost).
        if (MORE || skip + 2 > STAGES) ok = ok && wait_on(S.far_over, (uint32_t)it & 1u, abort_flag);
        k.skip(skip);
        uint32_t sp = 0;
        for (int j = 0; j <= walk.near && ok; ++j) {
          const uint32_t s = k.s;
          if (j < walk.near) {
            ok = filled() && (t == 0 || wait_on(S.s_free, (t - 1) & 1u, abort_flag));
            if (!ok) break;
            tc_fence_after();
            mma_scores(tmem, qd, kd0 + step * s);
            mma_scores(tmem + 64, gd, kd0 + step * s + vofs);
            tc_commit(S.s_full);
            if (j + 1 == walk.near) tc_commit(S.own_free);
            ++t;
            k.next();
          }
          if (j > 0) {
            ok = wait_on(S.w_full, (t - (j < walk.near ? 2u : 1u)) & 1u, abort_flag);
            if (!ok) break;
            tc_fence_after();
            mma_weights(tmem + 128, tmem + 192, 8, kd0 + step * sp, j > 1 ? 1u : from_far);
            mbar_arrive_n(S.empty + 8 * sp, SLOT_ARRIVALS - 1);
            tc_commit(S.empty + 8 * sp);
            tc_commit(j == walk.near ? S.acc_full : S.w_free);
          }
          sp = s;
        }
        k.next();              // the results' slot
        ok = ok && next_block<MORE>(S, P, it, at, abort_flag);
        fence_async_smem();
      }
    }
  } else {
    const int quarter = warp & 3, c = (warp >> 2) * COLS;    // this warp's lanes, and its share of a tile's 64 columns
    const int r = quarter * 32 + lane, rs = quarter * 32 + (warp >> 2) * 16;   // this thread's row; this warp's sixteen of the far tiles
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
    float* part = S.at<float>(S.part);                       // [PARTS][128] partial sums of delta
    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E);
    Ring<STAGES> k;
    uint32_t t = 0, frees = 0, leaving = 0;
    bool ok = true;
    // the copies that take a lane quarter's results away have read them: their slot may be filled again.  Asked a block later, when they have
    // long done so.
    auto results_gone = [&]() {
      bulk_wait_read();
      mbar_arrive(leaving);
    };
    // this row's log-sum-exp, on its way while the block before leaves; a block without successors fetches its share of the forward output
    // as well (through a slot it would wait behind the own rows)
    float nl;
    uint4 out_row[COLS / 8] = {};
    auto fetch_row = [&](const Place& p) {
      const int i = (P.blocks - 1 - p.block) * ROWS + r;
      nl = 0.f;
      if (i < P.seq) {
        if (!MORE) {
          const uint4* src = reinterpret_cast<const uint4*>(P.Out + ((int64_t)p.b * P.seq + i) * P.ldo + p.h * D + c);
#pragma unroll
          for (int e = 0; e < COLS / 8; ++e) out_row[e] = __ldg(src + e);
        }
        nl = __ldg(P.lse + ((int64_t)p.b * P.heads + p.h) * P.seq + i);
      }
    };
    fetch_row(at);
    for (int it = 0; ok; ++it) {
      const int h = at.h, b = at.b, q0 = (P.blocks - 1 - at.block) * ROWS, row0 = b * P.seq;
      const int i = q0 + r;
      const Walk<true> walk = MORE ? Walk<true>(q0, l, P.seq, P.magic) : first;
      const int far = FAR ? walk.far() : 0;
      // delta of this row: the threads of a row take COLS dimensions each
      const bool row_ok = i < P.seq;
      nl *= -LOG2E;
      if (it > 0 && c == 0 && lane == 0) results_gone();
      ok = wait_on(S.own_full, (uint32_t)it & 1u, abort_flag) && (!MORE || wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag));
      float del = 0.f;
#pragma unroll
      for (int p = 0; p < COLS / 8; ++p) {
        const uint4 o = MORE ? lds128(piece_addr(S.ring + k.s * SLOT_BYTES, r, c / 8 + p)) : out_row[p], g = lds128(piece_addr(S.own1, r, c / 8 + p));
        const uint32_t ow[4] = {o.x, o.y, o.z, o.w}, gw[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          del = fmaf(bf_lo(ow[e]), bf_lo(gw[e]), del);
          del = fmaf(bf_hi(ow[e]), bf_hi(gw[e]), del);
        }
      }
      if (MORE) {
        fence_async_smem();
        __syncwarp();
        if (lane == 0) mbar_arrive(S.empty + 8 * k.s);
        k.next();
      }
      part[c / COLS * ROWS + r] = del;
      ok = meet(S, quarter, 0u, lane, abort_flag) && ok;
      del = 0.f;
#pragma unroll
      for (int p = 0; p < PARTS; ++p) del += part[p * ROWS + r];
      if (c == 0 && row_ok) {
        const int64_t st = ((int64_t)b * P.heads + h) * P.seq + i;
        float* out = P.stat + (st / TS) * (2 * TS) + r % TS;   // st = r modulo 64
        out[0] = nl;
        out[TS] = -del;
      }
      // far tiles: warp = 16 rows of the block, with the keys in line with them
      if (far > 0) {
        float acc[8][4];
#pragma unroll
        for (int nb = 0; nb < 8; ++nb) acc[nb][0] = acc[nb][1] = acc[nb][2] = acc[nb][3] = 0.f;
        const int g = lane >> 2, tq = lane & 3, c0 = rs & 63;
        const float2 st0 = make_float2(__shfl_sync(0xffffffffu, nl, (rs & 31) + g), __shfl_sync(0xffffffffu, del, (rs & 31) + g));
        const float2 st1 = make_float2(__shfl_sync(0xffffffffu, nl, (rs & 31) + g + 8), __shfl_sync(0xffffffffu, del, (rs & 31) + g + 8));
        for (int f = walk.far_first(quarter >> 1); f < far; f += walk.far_step()) {
          Ring<STAGES> kf = k;
          kf.skip(f);
          ok = wait_on(S.full + 8 * kf.s, kf.lap & 1u, abort_flag);
          if (!ok) break;
          const uint32_t kt = S.ring + kf.s * SLOT_BYTES;
          float sc[2][4], dp[2][4];
          far_scores(sc, S.own0, rs, kt, c0, lane);
          far_scores(dp, S.own1, rs, kt + TILE_BYTES, c0, lane);
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float ds = 0.f;
              if (g + (e >> 1) * 8 == nb * 8 + 2 * tq + (e & 1)) {
                const float p = ex2(fmaf(sc[nb][e], SCALE_LOG2E, (e >> 1) ? st1.x : st0.x));
                ds = p * (dp[nb][e] - ((e >> 1) ? st1.y : st0.y));
              }
              sc[nb][e] = ds;
            }
          }
          far_accumulate(acc, sc, kt, c0, lane);
          far_release(S.empty + 8 * kf.s, lane);
        }
        k.skip(far);
        tmem_st_tiles(tmem + ((uint32_t)rs << 16) + 128u, acc);
        tmem_st_wait();                                      // ordered before the products by this warp's next arrivals
      }
      fence_async_smem();                                    // the own rows and the last answer have been read
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(S.own_free);
        mbar_arrive(S.far_over);
      }
      if (far > 0) ok = wait_on(S.far_over, (uint32_t)it & 1u, abort_flag) && ok;

      const uint64_t nl2 = pack2(nl, nl), ndel2 = pack2(-del, -del);
      const int i_lo = q0 + quarter * 32;                    // this warp's rows: i_lo .. i_lo + 31
      for (int j = 0; j < walk.near && ok; ++j, ++t) {
        ok = wait_on(S.s_full, t & 1u, abort_flag);
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
          ok = wait_on(S.w_free, frees & 1u, abort_flag);
          if (!ok) break;
          ++frees;
          tc_fence_after();
        }
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc) tmem_st8(t_row + (uint32_t)(192 + c / 2 + pc * 8), w[pc]);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(S.w_full);
      }
      k.skip(walk.near);
      const bool more = ok && next_block<MORE>(S, P, it, at, abort_flag);
      if (more) fetch_row(at);
      ok = ok && (!MORE || wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag)) && wait_on(S.acc_full, (uint32_t)it & 1u, abort_flag);
      tc_fence_after();
      const uint32_t res = MORE ? S.ring + k.s * SLOT_BYTES : S.own0;   // without successors the own rows have been read for good
      uint32_t v[PIECES][16];
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(128 + c + pc * 16), v[pc]);
#pragma unroll
      for (int pc = 0; pc < PIECES; ++pc) {
        tmem_ld16_wait(v[pc]);
        stage_row(res, r, c + pc * 16, v[pc], SCALE);
      }
      if (!MORE) {
        ok = meet(S, quarter, 1u, lane, abort_flag) && ok;
        if (ok && q0 + quarter * 32 < P.seq) write_rows(res, rs, P.dQ + ((int64_t)row0 + q0) * P.ldg + h * D, P.ldg, lane);
        break;
      }
      fence_async_smem();
      tc_fence_before();                                     // the accumulator has been read
      ok = meet(S, quarter, 1u, lane, abort_flag) && ok;
      tc_fence_after();
      if (c == 0) {
        if (lane == 0) {
          if (ok && q0 + quarter * 32 < P.seq) tma_store_2d(&tmD, res + (uint32_t)quarter * 32u * 128u, h * D, row0 + q0 + quarter * 32);
          bulk_commit();
          leaving = S.empty + 8 * k.s;
        }
      } else if (lane == 0) {
        mbar_arrive(S.empty + 8 * k.s);
      }
      k.next();
      ok = ok && more;
    }
    if (MORE && c == 0 && lane == 0) bulk_wait_read();       // shared memory outlives the copies
  }
  block_teardown(tmem, warp, abort_flag);
}

// ------------------------------------------------------------------------------------------- dK, dV
// Tensor memory: S^T in columns 0-63, dP^T 64-127, dK 128-191, dV 192-255; each warp writes P^T over the scores it has
// read (eight columns at its sixteen's start) and dS^T over its dP.
template <bool MORE, bool FAR>   // see mst_attention_tile.cuh
__global__ void __launch_bounds__(THREADS, 2)
attn_bwd_dkv_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                    const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmG, const __grid_constant__ CUtensorMap tmDK,
                    const __grid_constant__ CUtensorMap tmDV, const BwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const Smem S(smem_raw);
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = P.stride;
  if (warp == CW && lane < (MORE ? 6 : 4)) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : lane == 3 ? &tmG : lane == 4 ? &tmDK : &tmDV);
  const uint32_t tmem = block_setup(S, &holder, &abort_sh, warp);
  Place at = place((int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, P.blocks, P.heads, !MORE && P.blocks_first);   // early keys have the most tiles
  Walk<false> first(at.block * ROWS, l, P.seq, P.magic);
  if (!MORE) first.now();
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  if (warp == CW) {
    if (lane == 0) feed<false, 2, MORE>(S, P, at, first, &tmK, &tmV, &tmQ, &tmG, nullptr, abort_flag);
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t kd = smem_desc(S.own0, 16, 1024), vd = smem_desc(S.own1, 16, 1024), qd0 = smem_desc(S.ring, 16, 1024);
      const uint64_t step = SLOT_BYTES >> 4, gofs = TILE_BYTES >> 4;
      Ring<STAGES> k;
      uint32_t t = 0;   // near tiles so far
      bool ok = true;
      auto filled = [&]() { return wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag); };
      for (int it = 0; ok; ++it) {
        const Walk<false> walk = MORE ? Walk<false>(at.block * ROWS, l, P.seq, P.magic) : first;
        const uint32_t from_far = FAR && walk.far() > 0 ? 1u : 0u;
        ok = wait_on(S.own_full, (uint32_t)it & 1u, abort_flag);
        if (MORE || walk.far() + 1 > STAGES) ok = ok && wait_on(S.far_over, (uint32_t)it & 1u, abort_flag);   // as in dQ, for one tile
        k.skip(walk.far());
        ok = ok && filled();
        for (int j = 0; j < walk.near && ok; ++j, ++t) {
          const uint32_t s = k.s;
          const uint64_t qd = qd0 + step * s;
          tc_fence_after();
          // Everything executes in issue order, so the scores may overwrite the P of the tile before (its dV product is issued)
          // and dP its dS.  S goes ahead of the last tile's dK: the exponentials start while dK and dP are formed.
          if (j == 0) mma_scores(tmem, kd, qd);
          if (j == 0) tc_commit(S.s_full);
          mma_scores(tmem + 64, vd, qd + gofs);
          tc_commit(S.dp_full);
          if (j + 1 == walk.near) tc_commit(S.own_free);
          ok = wait_on(S.p_full, t & 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          mma_weights(tmem + 192, tmem, 16, qd + gofs, j > 0 ? 1u : from_far);
          k.next();
          if (j + 1 < walk.near) {
            ok = filled();
            if (!ok) break;
            tc_fence_after();
            mma_scores(tmem, kd, qd0 + step * k.s);
            tc_commit(S.s_full);
          }
          ok = wait_on(S.w_full, t & 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          mma_weights(tmem + 128, tmem + 64, 16, qd, j > 0 ? 1u : from_far);
          mbar_arrive_n(S.empty + 8 * s, SLOT_ARRIVALS - 1);
          tc_commit(S.empty + 8 * s);
          if (j + 1 == walk.near) tc_commit(S.acc_full);
        }
        k.skip(2);             // the results' slots
        ok = ok && next_block<MORE>(S, P, it, at, abort_flag);
        fence_async_smem();
      }
    }
  } else {
    const int quarter = warp & 3, c = (warp >> 2) * COLS;    // this warp's lanes, and its share of a tile's 64 columns
    const int r = quarter * 32 + lane, rs = quarter * 32 + (warp >> 2) * 16;   // this thread's row; this warp's sixteen of the far tiles
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16);
    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E);
    Ring<STAGES> k;
    uint32_t t = 0;
    bool ok = true;
    for (int it = 0; ok; ++it) {
      const int h = at.h, k0 = at.block * ROWS, row0 = at.b * P.seq;
      const int jk = k0 + r, j_lo = k0 + quarter * 32;       // this thread's key, this warp's: j_lo .. j_lo + 31
      const Walk<false> walk = MORE ? Walk<false>(k0, l, P.seq, P.magic) : first;
      const int far = FAR ? walk.far() : 0;
      if (it > 0 && c == 0 && lane == 0) {                   // the copies of the last results have read them, long since: their slots may be filled again
        bulk_wait_read();
        mbar_arrive(S.empty + 8 * ((k.s + STAGES - 2) % STAGES));
        mbar_arrive(S.empty + 8 * ((k.s + STAGES - 1) % STAGES));
      }
      ok = wait_on(S.own_full, (uint32_t)it & 1u, abort_flag);
      // far tiles: warp = 16 keys of the block, with the queries in line with them
      if (far > 0) {
        float acc_k[8][4], acc_v[8][4];
#pragma unroll
        for (int nb = 0; nb < 8; ++nb) {
          acc_k[nb][0] = acc_k[nb][1] = acc_k[nb][2] = acc_k[nb][3] = 0.f;
          acc_v[nb][0] = acc_v[nb][1] = acc_v[nb][2] = acc_v[nb][3] = 0.f;
        }
        const int g = lane >> 2, tq = lane & 3, c0 = rs & 63;
        for (int f = walk.far_first(quarter >> 1); f < far; f += walk.far_step()) {
          Ring<STAGES> kf = k;
          kf.skip(f);
          ok = wait_on(S.full + 8 * kf.s, kf.lap & 1u, abort_flag);
          if (!ok) break;
          const uint32_t qt = S.ring + kf.s * SLOT_BYTES;
          float st[2][4], dp[2][4];
          far_scores(st, S.own0, rs, qt, c0, lane);
          far_scores(dp, S.own1, rs, qt + TILE_BYTES, c0, lane);
#pragma unroll
          for (int nb = 0; nb < 2; ++nb) {
            const float* sq = S.at<float>(S.stat + kf.s * STAT_BYTES) + c0 + nb * 8 + 2 * tq;
            const float2 nl = *reinterpret_cast<const float2*>(sq), nd = *reinterpret_cast<const float2*>(sq + TS);
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              float p = 0.f, ds = 0.f;
              if (g + (e >> 1) * 8 == nb * 8 + 2 * tq + (e & 1)) {
                p = ex2(fmaf(st[nb][e], SCALE_LOG2E, (e & 1) ? nl.y : nl.x));
                ds = p * (dp[nb][e] + ((e & 1) ? nd.y : nd.x));
              }
              st[nb][e] = p;
              dp[nb][e] = ds;
            }
          }
          far_accumulate(acc_v, st, qt + TILE_BYTES, c0, lane);
          far_accumulate(acc_k, dp, qt, c0, lane);
          far_release(S.empty + 8 * kf.s, lane);
        }
        k.skip(far);
        tmem_st_tiles(tmem + ((uint32_t)rs << 16) + 128u, acc_k);
        tmem_st_tiles(tmem + ((uint32_t)rs << 16) + 192u, acc_v);
        tmem_st_wait();                                      // ordered before the products by this warp's next arrivals
      }
      fence_async_smem();                                    // the own rows and the last answer have been read
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(S.own_free);
        mbar_arrive(S.far_over);
      }
      if (far > 0) ok = wait_on(S.far_over, (uint32_t)it & 1u, abort_flag) && ok;
      for (int j = 0; j < walk.near && ok; ++j, ++t) {
        const uint32_t sa = S.stat + k.s * STAT_BYTES + (uint32_t)(c * 4);
        ok = wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag) &&   // the statistics have landed too
             wait_on(S.s_full, t & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
        uint32_t w[PIECES][8], st[PIECES][16];
        uint64_t p[PIECES][8];                               // P^T of this row, fp32 pairs
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(c + pc * 16), st[pc]);
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc) {
          const int q0 = walk.first + j * TS + c + pc * 16;  // the piece's queries: q0 .. q0 + 15
          tmem_ld16_wait(st[pc]);
          if (q0 + 15 >= j_lo && q0 - (j_lo + 31) <= l) {    // some pair is attended
#pragma unroll
            for (int e = 0; e < 4; ++e) {                    // statistics of four queries at a time
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
        ok = wait_on(S.dp_full, t & 1u, abort_flag);
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
        fence_async_smem();                                  // the statistics have been read
        __syncwarp();
        if (lane == 0) mbar_arrive(S.w_full);
        k.next();
      }
      ok = ok && wait_on(S.acc_full, (uint32_t)it & 1u, abort_flag);
      tc_fence_after();
      uint32_t at_slot[2];
#pragma unroll
      for (int which = 0; which < 2; ++which) {              // dK and dV, through a slot each
        ok = ok && (!MORE || wait_on(S.full + 8 * k.s, k.lap & 1u, abort_flag));
        at_slot[which] = MORE ? S.ring + k.s * SLOT_BYTES : which ? S.own1 : S.own0;
        k.next();
        uint32_t v[PIECES][16];
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc) tmem_ld16_nowait(t_row + (uint32_t)(128 + which * 64 + c + pc * 16), v[pc]);
#pragma unroll
        for (int pc = 0; pc < PIECES; ++pc) {
          tmem_ld16_wait(v[pc]);
          stage_row(at_slot[which], r, c + pc * 16, v[pc], which ? 1.f : SCALE);
        }
      }
      if (!MORE) {
        ok = meet(S, quarter, 0u, lane, abort_flag) && ok;
        if (ok && k0 + quarter * 32 < P.seq) {
          write_rows(at_slot[0], rs, P.dK + ((int64_t)row0 + k0) * P.ldg + h * D, P.ldg, lane);
          write_rows(at_slot[1], rs, P.dV + ((int64_t)row0 + k0) * P.ldg + h * D, P.ldg, lane);
        }
        break;
      }
      fence_async_smem();
      tc_fence_before();                                     // the accumulators have been read
      ok = meet(S, quarter, (uint32_t)it & 1u, lane, abort_flag) && ok;
      tc_fence_after();
      if (lane == 0) {
        if (c == 0) {
          if (ok && k0 + quarter * 32 < P.seq) {
            tma_store_2d(&tmDK, at_slot[0] + (uint32_t)quarter * 32u * 128u, h * D, row0 + k0 + quarter * 32);
            tma_store_2d(&tmDV, at_slot[1] + (uint32_t)quarter * 32u * 128u, h * D, row0 + k0 + quarter * 32);
          }
          bulk_commit();
        } else {
          mbar_arrive(S.empty + 8 * ((k.s + STAGES - 2) % STAGES));
          mbar_arrive(S.empty + 8 * ((k.s + STAGES - 1) % STAGES));
        }
      }
      ok = ok && next_block<MORE>(S, P, it, at, abort_flag);
    }
    if (MORE && c == 0 && lane == 0) bulk_wait_read();       // shared memory outlives the copies
  }
  block_teardown(tmem, warp, abort_flag);
}

struct Maps { CUtensorMap Q, K, V, G, O, dQ, dK, dV; };
template <bool MORE, bool FAR>
mst_status_t launch(dim3 grid, const Maps& m, const BwdParams& P, cudaStream_t s) {
  MST_SMEM_LIMIT((attn_bwd_dq_kernel<MORE, FAR>), SMEM_BYTES);
  MST_SMEM_LIMIT((attn_bwd_dkv_kernel<MORE, FAR>), SMEM_BYTES);
  MST_CUDA_TRY(mst_launch_overlapped(attn_bwd_dq_kernel<MORE, FAR>, grid, dim3(THREADS), SMEM_BYTES, s, m.Q, m.K, m.V, m.G, m.O, m.dQ, P));
  MST_CUDA_TRY(mst_launch_overlapped(attn_bwd_dkv_kernel<MORE, FAR>, grid, dim3(THREADS), SMEM_BYTES, s, m.Q, m.K, m.V, m.G, m.dK, m.dV, P));
  return MST_OK;
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
  const int blocks = (seq_len + ROWS - 1) / ROWS, l = stride < seq_len ? stride : seq_len;   // from there on the same pairs: all earlier positions
  const Form form = form_of(batch, heads, blocks, l, seq_len);
  Maps m = {};
  if (!tile_map(&m.Q, Q, rows, width, ld) || !tile_map(&m.K, K, rows, width, ld) || !tile_map(&m.V, V, rows, width, ld) ||
      !tile_map(&m.G, dOut, rows, width, lddo))
    return MST_ERR_SHAPE;
  if (form.more && (!tile_map(&m.O, Out, rows, width, ldo) || !tile_map(&m.dQ, dQ, rows, width, ldg, ROWS / 4) ||
                    !tile_map(&m.dK, dK, rows, width, ldg, ROWS / 4) || !tile_map(&m.dV, dV, rows, width, ldg, ROWS / 4)))
    return MST_ERR_SHAPE;
  void* ws = nullptr;
  MST_TRY(mst_workspace_kind(MST_WS_ATTENTION, 2 * sizeof(float) * (size_t)rows * heads, &ws));
  BwdParams P;
  P.Out = (const __nv_bfloat16*)Out;
  P.ldo = ldo;
  P.lse = lse; P.stat = (float*)ws;
  P.dQ = (__nv_bfloat16*)dQ; P.dK = (__nv_bfloat16*)dK; P.dV = (__nv_bfloat16*)dV;
  P.ldg = ldg;
  P.seq = seq_len; P.heads = heads; P.blocks = blocks; P.blocks_first = form.blocks_first;
  P.stride = l;
  P.magic = stride_magic(l, seq_len);
  const dim3 grid = place_grid(heads, batch, blocks, form.blocks_first);
  MST_TRY((form.more ? launch<true, true> : form.far ? launch<false, true> : launch<false, false>)(grid, m, P, s));
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}
