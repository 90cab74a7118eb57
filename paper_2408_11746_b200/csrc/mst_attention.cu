// Strided sparse self-attention, forward (Sec. 3.3):
//   Out[i] = sum_{j in S_i} P_ij v_j,   P = softmax over S_i of q_i . k_j / sqrt(d),
//   S_i = { j <= i : i - j < l  or  (i - j) mod l == 0 }, the same in every head.
// A block owns 128 queries of one (sequence, head).  It visits the far strided positions (i - 2l, i - 3l, ...) first, as tiles of which
// only the diagonal counts, and then walks 64-key tiles of the window (the tile that starts l back also holds the first strided key of
// every query).  When it is done it takes over a block that has not started (mst_attention_tile.cuh), whose operands are then on
// their way already.
// Roles of its ten warps:
//   warps 0-7  softmax: thread = query (tensor-memory lane), the two warps of a lane quarter take 32 of a tile's 64 keys each.
//              The two are softmaxes of their own - reference, sum and output accumulator, merged when the rows leave - so a tile
//              needs no exchange between them.  The reference follows the running maximum only when that has moved up by
//              more than 2^16 (fp32 sums and bf16 weights lose nothing by it), so accumulators are rescaled rarely.
//   warp 8     one lane feeds a four-slot ring by TMA;
//   warp 9     one lane issues tcgen05.mma: S = Q K^T (128 x 64) two tiles ahead, O_half += P V over the half's 32 keys, P read
//              from tensor memory where the softmax warps have written it over the scores.
// Tensor memory: scores in columns 0-63 and 64-127 (tiles alternate), the halves' outputs in 128-191 and 192-255.  256 columns
// and 83 KiB of shared memory: two blocks per SM, one's products and loads behind the other's softmax.
// The far tiles' softmax (two lanes a row, 16 rows a warp) is where the first half starts: reference and sum through shared memory, outputs in tensor memory.
// Results leave by TMA from a slot of the ring, or, in a block without successors, as whole rows from where the own rows were.
// Bound: the chain of a tile through its warps (scores, exponentials, weights: about 1000 clocks for a block, two of them at
// work on an SM).  16 x 1024 tokens, 12 heads, l = 256 50.2 -> 40 us,
// 8 x 1024, 16 heads, l = 128 35.5 -> 28.4 (one block after the other, heads last in the grid, far tiles at the end, on mma.sync).
#include <cuda.h>
#include <cuda_bf16.h>

#include "mst_attention_tile.cuh"
#include "mst_internal.cuh"

namespace {
using namespace mst_att;

constexpr int STAGES = 4;
constexpr int RING_BYTES = STAGES * SLOT_BYTES;
constexpr int STAT_FLOATS = 3 * 2 * ROWS;          // references and sums of the halves' softmaxes and of the far tiles'
constexpr int TMEM_COLS = 256;
constexpr float LAZY = 16.f;
// own rows, ring, statistics, answers, barriers: full and empty per stage, own_full, own_free, s_full[2], p_full[2], o_done, acc_full, next_full[2], pair[4], far_over
constexpr size_t SMEM_BYTES = 2 * TILE_BYTES + RING_BYTES + STAT_FLOATS * 4 + 32 + 16 * STAGES + 15 * 8 + 1024;

__device__ int g_attn_error = 0;

struct FwdParams {
  __nv_bfloat16* Out;
  int64_t ldo;
  float* lse;          // [batch, heads, seq] or NULL
  int seq, heads, stride, blocks, blocks_first;
  uint32_t magic;
};

__device__ __forceinline__ bool wait_on(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait(bar, parity, abort_flag, &g_attn_error);
}

// The exponents of a row are taken against m; a row that has seen nothing keeps m = -inf and takes them against 0
__device__ __forceinline__ float reference(float m) { return m == -INFINITY ? 0.f : m; }

template <bool MORE, bool FAR>   // see mst_attention_tile.cuh
__global__ void __launch_bounds__(THREADS, 2)
strided_attention_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                             const __grid_constant__ CUtensorMap tmV, const __grid_constant__ CUtensorMap tmO, const FwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t own = (smem_u32(smem_raw) + 1023u) & ~1023u, ring = own + 2 * TILE_BYTES, stat_a = ring + RING_BYTES;
  const uint32_t answers = stat_a + STAT_FLOATS * 4;
  const uint32_t full = answers + 32, empty = full + 8 * STAGES, own_full = empty + 8 * STAGES, own_free = own_full + 8,
                 s_full = own_free + 8, p_full = s_full + 16, o_done = p_full + 16, acc_full = o_done + 8, next_full = acc_full + 8,
                 pair0 = next_full + 16, far_over = pair0 + 32;
  unsigned char* base = smem_raw + (own - smem_u32(smem_raw));
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int l = P.stride;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full + 8 * s, 1);
      mbar_init(empty + 8 * s, SLOT_ARRIVALS);
    }
    mbar_init(own_full, 1);
    mbar_init(own_free, 1 + CW);
    for (int e = 0; e < 2; ++e) {
      mbar_init(s_full + 8 * e, 1);
      mbar_init(p_full + 8 * e, CW);       // one per buffer: a warp may be a tile ahead of another
      mbar_init(next_full + 8 * e, 1);
    }
    mbar_init(o_done, 1);
    mbar_init(acc_full, 1);
    for (int e = 0; e < 4; ++e) mbar_init(pair0 + 8 * e, 2);
    mbar_init(far_over, CW);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == CW && lane < (MORE ? 4 : 3)) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : lane == 2 ? &tmV : &tmO);
  if (warp == CW + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&holder)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = holder;
  Place at = place((int)blockIdx.x, (int)blockIdx.y, (int)blockIdx.z, P.blocks, P.heads, !MORE && P.blocks_first);
  Walk<true> first((P.blocks - 1 - at.block) * ROWS, l, P.seq, P.magic);
  if (!MORE) first.now();
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  Ring<STAGES> k;
  // the next block, if there is one (block `it` of this one's life is at its end)
  auto next = [&](int it) { return MORE && wait_on(next_full + 8 * (it & 1), (uint32_t)(it >> 1) & 1u, abort_flag) && taken_over(answers + 16 * (it & 1), at, P.blocks, P.heads); };
  auto next_fenced = [&](int it) {   // for the lanes that have no other fence ahead of their part in the own rows' release
    const bool more = next(it);
    fence_async_smem();
    return more;
  };

  if (warp == CW) {
    if (lane == 0) {
      bool ok = true;
      auto slot = [&]() { return k.lap == 0 || wait_on(empty + 8 * k.s, (k.lap - 1) & 1u, abort_flag); };
      for (int it = 0; ok; ++it) {
        const int col = at.h * D, row0 = at.b * P.seq, q0 = (P.blocks - 1 - at.block) * ROWS;   // late queries have the most tiles
        const Walk<true> walk = MORE ? Walk<true>(q0, l, P.seq, P.magic) : first;
        if (it > 0 && !wait_on(own_free, (uint32_t)(it - 1) & 1u, abort_flag)) break;
        mbar_expect_tx(own_full, 2 * TILE_BYTES);
        tma_load_2d(own, &tmQ, col, row0 + q0, own_full);
        tma_load_2d(own + TILE_BYTES, &tmQ, col, row0 + q0 + TS, own_full);
        if (MORE) take_over(answers + 16 * (it & 1), next_full + 8 * (it & 1));
        for (int j = 0; j < walk.total && ok; ++j) {
          ok = slot();
          if (!ok) break;
          const uint32_t dst = ring + k.s * SLOT_BYTES, bar = full + 8 * k.s;
          mbar_expect_tx(bar, 2 * TILE_BYTES);
          tma_load_2d(dst, &tmK, col, row0 + walk.start(j), bar);
          tma_load_2d(dst + TILE_BYTES, &tmV, col, row0 + walk.start(j), bar);
          k.next();
        }
        ok = ok && MORE && slot();       // a slot for the results
        if (!ok) break;
        mbar_arrive(full + 8 * k.s);
        k.next();
        ok = next_fenced(it);
      }
    }
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t qd = smem_desc(own, 16, 1024), kd0 = smem_desc(ring, 16, 1024);
      const uint64_t step = SLOT_BYTES >> 4, vofs = TILE_BYTES >> 4;
      uint32_t t = 0;   // near tiles so far: tile t has its scores in buffer t % 2
      bool ok = true;
      auto filled = [&]() { return wait_on(full + 8 * k.s, k.lap & 1u, abort_flag); };
      for (int it = 0; ok; ++it) {
        const Walk<true> walk = MORE ? Walk<true>((P.blocks - 1 - at.block) * ROWS, l, P.seq, P.magic) : first;
        const int near = walk.near;
        const uint32_t from_far = FAR && walk.far() > 0 ? 1u : 0u;
        ok = wait_on(own_full, (uint32_t)it & 1u, abort_flag);
        // in a block without successors the first two tiles' scores need not wait for the far tiles where their slots are filled for the
        // first time (see dQ)
        if (MORE || walk.far() + 2 > STAGES) ok = ok && wait_on(far_over, (uint32_t)it & 1u, abort_flag);
        k.skip(walk.far());
        Ring<STAGES> kv = k;             // the tile whose weights are ready next
        // scores of tile j, in issue order behind the product that read the weights of the tile two before there
        auto scores = [&](int j) {
          if (!filled()) return false;
          tc_fence_after();
          mma_scores(tmem + ((t + (uint32_t)j) & 1u) * 64u, qd, kd0 + step * k.s);
          tc_commit(s_full + 8 * ((t + (uint32_t)j) & 1u));
          if (j + 1 == near) tc_commit(own_free);
          k.next();
          return true;
        };
        ok = ok && scores(0);
        if (ok && near > 1) ok = scores(1);
        for (int j = 0; j < near && ok; ++j) {
          const uint32_t tj = t + (uint32_t)j;
          ok = wait_on(p_full + 8 * (tj & 1u), (tj >> 1) & 1u, abort_flag);
          if (!ok) break;
          tc_fence_after();
          const uint32_t p = tmem + (tj & 1u) * 64u;
          const uint64_t vd = kd0 + step * kv.s + vofs;
#pragma unroll
          for (int ks = 0; ks < 4; ++ks)   // 16 keys each: two of the first half's 32, two of the second's
            tc_mma_ts(tmem + 128 + (uint32_t)(ks >> 1) * 64u, p + (uint32_t)((ks >> 1) * 32 + (ks & 1) * 8), vd + (uint64_t)(ks * ((16 * 128) >> 4)),
                      IDESC_MN, (j > 0 || (ks & 1)) ? 1u : ks == 0 ? from_far : 0u);
          mbar_arrive_n(empty + 8 * kv.s, SLOT_ARRIVALS - 1);
          tc_commit(empty + 8 * kv.s);
          tc_commit(o_done);
          if (j + 1 == near) tc_commit(acc_full);
          kv.next();
          if (j + 2 < near) ok = scores(j + 2);
        }
        t += (uint32_t)near;
        k.next();                        // the results' slot
        ok = ok && next_fenced(it);
      }
    }
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const int r = quarter * 32 + lane, rs = quarter * 32 + half * 16;   // this thread's row; this warp's sixteen of the far tiles
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16), t_out = t_row + 128u + (uint32_t)half * 64u;
    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E);
    float* stat = reinterpret_cast<float*>(base + (stat_a - own));   // [3][2][128]
    uint32_t t = 0, pairs = 0, leaving = 0;
    bool ok = true;
    // the copies that take a lane quarter's results away have read them: their slot may be filled again.  Asked a block later, when they have
    // long done so.
    auto results_gone = [&]() {
      bulk_wait_read();
      mbar_arrive(leaving);
    };
    // the two warps of a lane quarter meet
    auto meet = [&]() {
      __syncwarp();
      if (lane == 0) mbar_arrive(pair0 + 8 * quarter);
      const bool met = wait_on(pair0 + 8 * quarter, pairs & 1u, abort_flag);
      ++pairs;
      return met;
    };
    for (int it = 0; ok; ++it) {
      const int h = at.h, b = at.b, q0 = (P.blocks - 1 - at.block) * ROWS, row0 = b * P.seq;
      const int i = q0 + r, i_lo = q0 + quarter * 32;        // this thread's query, this warp's: i_lo .. i_lo + 31
      const Walk<true> walk = MORE ? Walk<true>(q0, l, P.seq, P.magic) : first;
      const int far = FAR ? walk.far() : 0;
      float m = -INFINITY;                                   // reference of this half's softmax, base 2
      uint64_t sum2 = 0ULL;
      ok = wait_on(own_full, (uint32_t)it & 1u, abort_flag);
      if (it > 0 && half == 0 && lane == 0) results_gone();
      // far tiles: a softmax of their own, which the first half goes on with
      if (far > 0) {
        const FarRow mine = far_row(own, rs + (lane & 15), lane);
        float acc[32], fm = -INFINITY, fs = 0.f;
#pragma unroll
        for (int e = 0; e < 32; ++e) acc[e] = 0.f;
        for (int f = walk.far_first(quarter >> 1); f < far; f += walk.far_step()) {
          Ring<STAGES> kf = k;
          kf.skip(f);
          ok = wait_on(full + 8 * kf.s, kf.lap & 1u, abort_flag);
          if (!ok) break;
          const uint32_t kt = ring + kf.s * SLOT_BYTES;
          const int row = (rs + (lane & 15)) & (TS - 1);
          const FarRow v = far_row(kt + TILE_BYTES, row, lane);
          const float x = far_dot(mine, far_row(kt, row, lane)) * SCALE_LOG2E;
          const bool up = x > fm + LAZY;
          if (__any_sync(0xffffffffu, up)) {
            const float c = up ? ex2(fm - x) : 1.f;
            if (up) fm = x;
            fs *= c;
#pragma unroll
            for (int e = 0; e < 32; ++e) acc[e] *= c;
          }
          const float w = ex2(x - reference(fm));
          fs += w;
          far_add(acc, w, v);
          far_release(empty + 8 * kf.s, lane);
        }
        k.skip(far);
        far_start_sums(tmem + ((uint32_t)rs << 16) + 128u, acc);
        if (lane < 16) {
          stat[4 * ROWS + rs + lane] = fm;
          stat[5 * ROWS + rs + lane] = fs;
        }
        tmem_st_wait();
        tc_fence_before();
      }
      fence_async_smem();                                    // the own rows and the last answer have been read
      __syncwarp();
      if (lane == 0) {
        mbar_arrive(own_free);
        mbar_arrive(far_over);
      }
      if (far > 0) {
        ok = wait_on(far_over, (uint32_t)it & 1u, abort_flag) && ok;
        tc_fence_after();
        if (half == 0) {
          m = stat[4 * ROWS + r];
          sum2 = pack2(stat[5 * ROWS + r], 0.f);
        }
      }
      for (int j = 0; j < walk.near && ok; ++j, ++t) {
        const int k0 = walk.first + j * TS + half * 32;      // this warp's keys: k0 .. k0 + 31
        ok = wait_on(s_full + 8 * (t & 1u), (t >> 1) & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const uint32_t t_s = t_row + (t & 1u) * 64u + (uint32_t)half * 32u;
        uint32_t w[16];
        if (i_lo + 31 >= k0 && i_lo - (k0 + 31) <= l) {      // some pair is attended
          uint32_t s[32];
          tmem_ld32(t_s, s);
          if (!(i_lo >= k0 + 31 && i_lo + 31 - k0 <= l)) {   // some pair is not
            const int back0 = i - k0;
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if ((unsigned)(back0 - e) > (unsigned)l) s[e] = 0xFF800000u;   // -inf
          }
          float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
          for (int e = 0; e < 32; e += 2) mx[(e >> 1) & 3] = fmaxf(mx[(e >> 1) & 3], fmaxf(__uint_as_float(s[e]), __uint_as_float(s[e + 1])));
          const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * SCALE_LOG2E;
          const bool up = top > m + LAZY;                    // a first key (m = -inf) always moves the reference
          if (__any_sync(0xffffffffu, up)) {
            const float c = up ? ex2(m - top) : 1.f;         // 0 where nothing has been summed yet
            const bool summed = up && m != -INFINITY;
            if (up) m = top;
            sum2 = mul2(sum2, pack2(c, c));
            if (__any_sync(0xffffffffu, summed)) {           // this half's outputs so far, once the tile before has been added
              ok = j == 0 || wait_on(o_done, (t - 1) & 1u, abort_flag);   // the first tile: sums of the far tiles
              if (!ok) break;
              tc_fence_after();
#pragma unroll 1
              for (int g = 0; g < 64; g += 16) {
                uint32_t v[16];
                tmem_ld16_nowait(t_out + (uint32_t)g, v);
                tmem_ld16_wait(v);
                uint32_t lo[8], hi[8];
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  lo[e] = __float_as_uint(__uint_as_float(v[e]) * c);
                  hi[e] = __float_as_uint(__uint_as_float(v[e + 8]) * c);
                }
                tmem_st8(t_out + (uint32_t)g, lo);
                tmem_st8(t_out + (uint32_t)(g + 8), hi);
              }
            }
          }
          const float nm = -reference(m);
          const uint64_t nm2 = pack2(nm, nm);
          uint64_t part[2] = {0ULL, 0ULL};
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const uint64_t p = ex2_2(fma2(pack2(s[2 * e], s[2 * e + 1]), scale2, nm2));
            part[e & 1] = add2(part[e & 1], p);
            w[e] = pack_bf16_2(p);
          }
          sum2 = add2(sum2, add2(part[0], part[1]));
        } else {
#pragma unroll
          for (int e = 0; e < 16; ++e) w[e] = 0u;
        }
        tmem_st16(t_s, w);
        tmem_st_wait();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(p_full + 8 * (t & 1u));
      }
      k.skip(walk.near);
      // the two softmaxes of row r meet: weights 2^(m_k - m) / sum
      float s_lo, s_hi;
      unpack2(sum2, s_lo, s_hi);
      stat[half * 2 * ROWS + r] = m;
      stat[half * 2 * ROWS + ROWS + r] = s_lo + s_hi;
      ok = meet() && ok;
      const float m0 = stat[r], m1 = stat[2 * ROWS + r];
      const float mm = fmaxf(m0, m1);                        // finite: a query attends to itself
      float a0 = ex2(m0 - mm), a1 = ex2(m1 - mm);
      const float total = fmaf(a0, stat[ROWS + r], a1 * stat[3 * ROWS + r]);
      const float inv = 1.f / total;
      a0 *= inv;
      a1 *= inv;
      ok = ok && (!MORE || wait_on(full + 8 * k.s, k.lap & 1u, abort_flag)) && wait_on(acc_full, (uint32_t)it & 1u, abort_flag);
      tc_fence_after();
      if (P.lse && half == 0 && ok) P.lse[((int64_t)b * P.heads + h) * P.seq + i] = (mm + log2f(total)) * 0.6931471805599453f;
      const uint32_t res = MORE ? ring + k.s * SLOT_BYTES : own;   // without successors the own rows have been read for good
#pragma unroll
      for (int pc = 0; pc < 2; ++pc) {
        const int c = half * 32 + pc * 16;
        uint32_t u[16], v[16];
        tmem_ld16_nowait(t_row + 128u + (uint32_t)c, u);
        tmem_ld16_nowait(t_row + 192u + (uint32_t)c, v);
        tmem_ld16_wait(u);
        tmem_ld16_wait(v);
#pragma unroll
        for (int e = 0; e < 16; ++e) u[e] = __float_as_uint(fmaf(a0, __uint_as_float(u[e]), a1 * __uint_as_float(v[e])));
        stage_row(res, r, c, u, 1.f);
      }
      if (!MORE) {
        ok = meet() && ok;
        if (ok) write_rows(res, rs, P.Out + ((int64_t)row0 + q0) * P.ldo + h * D, P.ldo, lane);
        break;
      }
      fence_async_smem();
      tc_fence_before();                                     // the accumulators have been read
      ok = meet() && ok;
      tc_fence_after();
      if (half == 0) {
        if (lane == 0) {
          if (ok) tma_store_2d(&tmO, res + (uint32_t)quarter * 32u * 128u, h * D, row0 + q0 + quarter * 32);
          bulk_commit();
          leaving = empty + 8 * k.s;
        }
      } else if (lane == 0) {
        mbar_arrive(empty + 8 * k.s);
      }
      k.next();
      ok = ok && next(it);
    }
    if (MORE && half == 0 && lane == 0) bulk_wait_read();    // shared memory outlives the copies
  }
  if (*abort_flag) {
    for (int t = 0; t < 2000; ++t) __nanosleep(1000);   // let copies and products in flight land
  }
  tc_fence_before();
  __syncthreads();
  if (warp == CW + 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TMEM_COLS) : "memory");
  }
}

template <bool MORE, bool FAR>
mst_status_t launch(dim3 grid, const CUtensorMap& tmQ, const CUtensorMap& tmK, const CUtensorMap& tmV, const CUtensorMap& tmO, const FwdParams& P,
                    cudaStream_t s) {
  MST_SMEM_LIMIT((strided_attention_fwd_kernel<MORE, FAR>), SMEM_BYTES);
  MST_CUDA_TRY(mst_launch_overlapped(strided_attention_fwd_kernel<MORE, FAR>, grid, dim3(THREADS), SMEM_BYTES, s, tmQ, tmK, tmV, tmO, P));
  return MST_OK;
}

}  // namespace

mst_status_t mst_attention_error_flags(int32_t* flags) {
  int v = 0;
  MST_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_attn_error, sizeof(int)));
  int32_t bwd = 0;
  MST_TRY(mst_attention_bwd_error_flags(&bwd));
  *flags = v | bwd;
  return MST_OK;
}

extern "C" mst_status_t mst_strided_attention_fwd(const void* Q, const void* K, const void* V, int64_t ld, int32_t batch,
                                                  int32_t seq_len, int32_t heads, int32_t head_dim, int32_t stride,
                                                  void* Out, int64_t ldo, float* lse, mst_stream_t stream) {
  if (!Q || !K || !V || !Out || batch < 0 || seq_len <= 0 || heads <= 0) return MST_ERR_INVALID_ARG;
  if (head_dim != D || seq_len % ROWS != 0 || stride <= 0 || stride % TS != 0) return MST_ERR_SHAPE;
  const int64_t width = (int64_t)heads * D;
  if (ld < width || ldo < width || ld % 8 != 0 || ldo % 8 != 0) return MST_ERR_SHAPE;
  if (((reinterpret_cast<uintptr_t>(Q) | reinterpret_cast<uintptr_t>(K) | reinterpret_cast<uintptr_t>(V) |
        reinterpret_cast<uintptr_t>(Out)) & 15u) != 0)
    return MST_ERR_SHAPE;
  if (batch == 0) return MST_OK;
  const int64_t rows = (int64_t)batch * seq_len;
  if (rows > 0x7FFFFFFF || heads > 65535 || batch > 65535) return MST_ERR_SHAPE;
  FwdParams P;
  P.Out = (__nv_bfloat16*)Out;
  P.ldo = ldo;
  P.lse = lse;
  P.seq = seq_len; P.heads = heads; P.blocks = seq_len / ROWS;
  P.stride = stride < seq_len ? stride : seq_len;   // from there on the same pairs: all earlier positions
  P.magic = stride_magic(P.stride, seq_len);
  const Form form = form_of(batch, heads, P.blocks, P.stride, seq_len);
  P.blocks_first = form.blocks_first;
  CUtensorMap tmQ, tmK, tmV, tmO = {};
  if (!tile_map(&tmQ, Q, rows, width, ld) || !tile_map(&tmK, K, rows, width, ld) || !tile_map(&tmV, V, rows, width, ld) ||
      (form.more && !tile_map(&tmO, Out, rows, width, ldo, ROWS / 4)))
    return MST_ERR_SHAPE;
  const dim3 grid = place_grid(heads, batch, P.blocks, form.blocks_first);
  MST_TRY((form.more ? launch<true, true> : form.far ? launch<false, true> : launch<false, false>)(grid, tmQ, tmK, tmV, tmO, P, (cudaStream_t)stream));
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}
