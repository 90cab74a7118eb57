// Strided sparse self-attention, forward (Sec. 3.3):
//   Out[i] = sum_{j in S_i} P_ij v_j,   P = softmax over S_i of q_i . k_j / sqrt(d),
//   S_i = { j <= i : i - j < l  or  (i - j) mod l == 0 }, the same in every head.
// A block owns 128 queries of one (sequence, head) and walks 64-key tiles of their window (the tile that starts l back also holds the
// first strided key of every query), then the far strided positions (i - 2l, i - 3l, ...) as tiles of which only the diagonal counts.
// Roles of its ten warps:
//   warps 0-7  softmax: thread = query (tensor-memory lane), the two warps of a lane quarter take 32 of a tile's 64 keys each.
//              The two are softmaxes of their own - reference, sum and output accumulator, merged when the rows leave - so a tile
//              needs no exchange between them.  The reference follows the running maximum only when that has moved up by
//              more than 2^16 (fp32 sums and bf16 weights lose nothing by it), so accumulators are rescaled rarely.
//   warp 8     one lane feeds a four-tile ring by TMA;
//   warp 9     one lane issues tcgen05.mma: S = Q K^T (128 x 64) two tiles ahead, O_half += P V over the half's 32 keys, P read
//              from tensor memory where the softmax warps have written it over the scores.
// Tensor memory: scores in columns 0-63 and 64-127 (tiles alternate), the halves' outputs in 128-191 and 192-255.  256 columns
// and 82 KiB of shared memory: two blocks per SM, one's products and loads behind the other's softmax.
// Far tiles are warp-level mma.sync products of 16 rows each with a softmax of their own, the third partial of the merge.
// Measured: 16 x 1024 tokens, 12 heads, l = 256 50 us, 8 x 1024, 16 heads, l = 128 35.5 us; the whole-window kernel (one tile per SM, S single)
// before took 67 us at l = 256, the mma.sync one 44 us at l = 128.
#include <cuda.h>
#include <cuda_bf16.h>

#include "mst_attention_tile.cuh"
#include "mst_internal.cuh"

namespace {
using namespace mst_att;

constexpr int CW = 8;                              // softmax warps
constexpr int THREADS = 32 * (CW + 2);
constexpr int STAGES = 4;
constexpr int RING_BYTES = STAGES * 2 * TILE_BYTES;
constexpr int STAT_FLOATS = 3 * 2 * ROWS;          // the three partial softmaxes' references and sums
constexpr int TMEM_COLS = 256;
constexpr float LAZY = 16.f;
// own rows, ring, statistics, barriers: full, empty, far_done per stage, own_full, s_full[2], p_full[2], o_done, acc_full
constexpr size_t SMEM_BYTES = 2 * TILE_BYTES + RING_BYTES + STAT_FLOATS * 4 + 24 * STAGES + 56 + 1024;
static_assert(ROWS * LDF * 4 + ROWS * LDO * 2 <= RING_BYTES, "the staged far sums and the staged results must fit the ring");

__device__ int g_attn_error = 0;

struct FwdParams {
  __nv_bfloat16* Out;
  int64_t ldo;
  float* lse;          // [batch, heads, seq] or NULL
  int seq, heads, stride;
  uint32_t magic;
};

__device__ __forceinline__ bool wait_on(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mbar_wait(bar, parity, abort_flag, &g_attn_error);
}

// The exponents of a row are taken against m; a row that has seen nothing keeps m = -inf and takes them against 0
__device__ __forceinline__ float reference(float m) { return m == -INFINITY ? 0.f : m; }

__global__ void __launch_bounds__(THREADS, 2)
strided_attention_fwd_kernel(const __grid_constant__ CUtensorMap tmQ, const __grid_constant__ CUtensorMap tmK,
                             const __grid_constant__ CUtensorMap tmV, const FwdParams P) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t own = (smem_u32(smem_raw) + 1023u) & ~1023u, ring = own + 2 * TILE_BYTES, stat_a = ring + RING_BYTES;
  const uint32_t full = stat_a + STAT_FLOATS * 4, empty = full + 8 * STAGES, far_done = empty + 8 * STAGES, own_full = far_done + 8 * STAGES,
                 s_full = own_full + 8, p_full = s_full + 16, o_done = p_full + 16, acc_full = o_done + 8;
  unsigned char* base = smem_raw + (own - smem_u32(smem_raw));
  __shared__ uint32_t holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int h = blockIdx.y, b = blockIdx.z, q0 = ((int)gridDim.x - 1 - (int)blockIdx.x) * ROWS, l = P.stride;   // late queries have the most tiles
  const int row0 = b * P.seq;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full + 8 * s, 1);
      mbar_init(empty + 8 * s, 1);
      mbar_init(far_done + 8 * s, CW / 2);
    }
    mbar_init(own_full, 1);
    mbar_init(s_full, 1);
    mbar_init(s_full + 8, 1);
    mbar_init(p_full, CW);       // one per buffer: a warp may be a tile ahead of another
    mbar_init(p_full + 8, CW);
    mbar_init(o_done, 1);
    mbar_init(acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == CW && lane < 3) prefetch_map(lane == 0 ? &tmQ : lane == 1 ? &tmK : &tmV);
  if (warp == CW + 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&holder)), "r"(TMEM_COLS) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = holder;
  const Walk<true> walk(q0, l, P.seq, P.magic);
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  if (warp == CW) {
    if (lane == 0) {
      const int col = h * D;
      mbar_expect_tx(own_full, 2 * TILE_BYTES);
      tma_load_2d(own, &tmQ, col, row0 + q0, own_full);
      tma_load_2d(own + TILE_BYTES, &tmQ, col, row0 + q0 + TS, own_full);
      feed_ring<STAGES>(walk, ring, full, empty, far_done, [&](int s, int at, uint32_t dst, uint32_t bar) {
        mbar_expect_tx(bar, 2 * TILE_BYTES);
        tma_load_2d(dst, &tmK, col, row0 + at, bar);
        tma_load_2d(dst + TILE_BYTES, &tmV, col, row0 + at, bar);
      }, [&](uint32_t bar, uint32_t parity) { return wait_on(bar, parity, abort_flag); });
    }
  } else if (warp == CW + 1) {
    if (lane == 0) {
      const uint64_t qd = smem_desc(own, 16, 1024), kd0 = smem_desc(ring, 16, 1024);
      const uint64_t step = (2 * TILE_BYTES) >> 4, vofs = TILE_BYTES >> 4;
      bool ok = wait_on(own_full, 0, abort_flag);
      // scores of tile j into buffer j % 2, in issue order behind the product that read P of tile j - 2 there
      auto scores = [&](int j) {
        const int s = j % STAGES;
        if (!wait_on(full + 8 * s, (uint32_t)(j / STAGES) & 1u, abort_flag)) return false;
        tc_fence_after();
        mma_scores(tmem + (uint32_t)(j & 1) * 64u, qd, kd0 + step * (uint32_t)s);
        tc_commit(s_full + 8 * (j & 1));
        return true;
      };
      if (ok) ok = scores(0);
      if (ok && walk.near > 1) ok = scores(1);
      for (int j = 0; j < walk.near && ok; ++j) {
        ok = wait_on(p_full + 8 * (j & 1), (uint32_t)(j >> 1) & 1u, abort_flag);
        if (!ok) break;
        tc_fence_after();
        const int s = j % STAGES;
        const uint32_t p = tmem + (uint32_t)(j & 1) * 64u;
        const uint64_t vd = kd0 + step * (uint32_t)s + vofs;
#pragma unroll
        for (int ks = 0; ks < 4; ++ks)   // 16 keys each: two of the first half's 32, two of the second's
          tc_mma_ts(tmem + 128 + (uint32_t)(ks >> 1) * 64u, p + (uint32_t)((ks >> 1) * 32 + (ks & 1) * 8), vd + (uint64_t)(ks * ((16 * 128) >> 4)),
                    IDESC_MN, (j > 0 || (ks & 1)) ? 1u : 0u);
        tc_commit(empty + 8 * s);
        tc_commit(o_done);
        if (j + 1 == walk.near) tc_commit(acc_full);
        if (j + 2 < walk.near) ok = scores(j + 2);
      }
    }
  } else {
    const int quarter = warp & 3, half = warp >> 2;
    const int r = quarter * 32 + lane, i = q0 + r;
    const int i_lo = q0 + quarter * 32;                      // this warp's queries: i_lo .. i_lo + 31
    const uint32_t t_row = tmem + ((uint32_t)(quarter * 32) << 16), t_out = t_row + 128u + (uint32_t)half * 64u;
    const uint64_t scale2 = pack2(SCALE_LOG2E, SCALE_LOG2E);
    float m = -INFINITY;                                     // reference of this half's softmax, base 2
    uint64_t sum2 = 0ULL;
    bool ok = true;
    for (int j = 0; j < walk.near && ok; ++j) {
      const int k0 = walk.first + j * TS + half * 32;        // this warp's keys: k0 .. k0 + 31
      ok = wait_on(s_full + 8 * (j & 1), (uint32_t)(j >> 1) & 1u, abort_flag);
      if (!ok) break;
      tc_fence_after();
      const uint32_t t_s = t_row + (uint32_t)((j & 1) * 64 + half * 32);
      uint32_t w[16];
      if (i_lo + 31 >= k0 && i_lo - (k0 + 31) <= l) {        // some pair is attended
        uint32_t s[32];
        tmem_ld32(t_s, s);
        if (!(i_lo >= k0 + 31 && i_lo + 31 - k0 <= l)) {     // some pair is not
          const int back0 = i - k0;
#pragma unroll
          for (int e = 0; e < 32; ++e)
            if ((unsigned)(back0 - e) > (unsigned)l) s[e] = 0xFF800000u;   // -inf
        }
        float mx[4] = {-INFINITY, -INFINITY, -INFINITY, -INFINITY};
#pragma unroll
        for (int e = 0; e < 32; e += 2) mx[(e >> 1) & 3] = fmaxf(mx[(e >> 1) & 3], fmaxf(__uint_as_float(s[e]), __uint_as_float(s[e + 1])));
        const float top = fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])) * SCALE_LOG2E;
        const bool up = top > m + LAZY;                      // a first key (m = -inf) always moves the reference
        if (__any_sync(0xffffffffu, up)) {
          const float c = up ? ex2(m - top) : 1.f;           // 0 where nothing has been summed yet
          const bool summed = up && m != -INFINITY;
          if (up) m = top;
          sum2 = mul2(sum2, pack2(c, c));
          if (__any_sync(0xffffffffu, summed)) {             // this half's outputs so far, once the tile before has been added
            ok = wait_on(o_done, (uint32_t)(j - 1) & 1u, abort_flag);
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
      if (lane == 0) mbar_arrive(p_full + 8 * (j & 1));
    }
    float s_lo, s_hi;
    unpack2(sum2, s_lo, s_hi);
    float* stat = reinterpret_cast<float*>(base + (stat_a - own));   // [3][2][128]
    stat[half * 2 * ROWS + r] = m;
    stat[half * 2 * ROWS + ROWS + r] = s_lo + s_hi;

    // far tiles: warp = 16 rows of the block, with the keys in line with them
    const int far = walk.far0 + walk.far1, rs = warp * 16;
    float acc[8][4];
#pragma unroll
    for (int nb = 0; nb < 8; ++nb) acc[nb][0] = acc[nb][1] = acc[nb][2] = acc[nb][3] = 0.f;
    if (far > 0) {
      const int g = lane >> 2, t = lane & 3, c0 = rs & 63;
      float fm[2] = {-INFINITY, -INFINITY}, fs[2] = {0.f, 0.f};   // rows rs + g and rs + g + 8; sums: this lane's columns only
      const int step = walk.far_step();
      for (int place = walk.near + walk.far_first(rs >> 6); place < walk.total; place += step) {
        const int s = place % STAGES;
        ok = wait_on(full + 8 * s, (uint32_t)(place / STAGES) & 1u, abort_flag);
        if (!ok) break;
        const uint32_t kt = ring + s * 2 * TILE_BYTES;
        float x[2][4];
        far_scores(x, own, rs, kt, c0, lane);
#pragma unroll
        for (int rr = 0; rr < 2; ++rr) {
          float v = -INFINITY;
#pragma unroll
          for (int nb = 0; nb < 2; ++nb)
#pragma unroll
            for (int e = 2 * rr; e < 2 * rr + 2; ++e) {
              if (g + rr * 8 != nb * 8 + 2 * t + (e & 1)) x[nb][e] = -INFINITY;
              v = fmaxf(v, x[nb][e]);
            }
          v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 1));
          v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 2)) * SCALE_LOG2E;
          if (v > fm[rr] + LAZY) {
            const float c = ex2(fm[rr] - v);
            fm[rr] = v;
            fs[rr] *= c;
#pragma unroll
            for (int nb = 0; nb < 8; ++nb) {
              acc[nb][2 * rr] *= c;
              acc[nb][2 * rr + 1] *= c;
            }
          }
          const float nm = -reference(fm[rr]);
#pragma unroll
          for (int nb = 0; nb < 2; ++nb)
#pragma unroll
            for (int e = 2 * rr; e < 2 * rr + 2; ++e) {
              x[nb][e] = ex2(fmaf(x[nb][e], SCALE_LOG2E, nm));
              fs[rr] += x[nb][e];
            }
        }
        far_accumulate<4>(acc, x, kt + TILE_BYTES, c0, 0, lane);
        far_release(far_done + 8 * s, lane);
      }
#pragma unroll
      for (int rr = 0; rr < 2; ++rr) {
        fs[rr] += __shfl_xor_sync(0xffffffffu, fs[rr], 1);
        fs[rr] += __shfl_xor_sync(0xffffffffu, fs[rr], 2);
        if (t == 0) {
          stat[4 * ROWS + rs + g + rr * 8] = fm[rr];
          stat[5 * ROWS + rs + g + rr * 8] = fs[rr];
        }
      }
    }
    ok = ok && wait_on(acc_full, 0, abort_flag);
    tc_fence_after();
    compute_sync<32 * CW>();   // every tile has been consumed: the ring takes the far sums and the results
    float* sums = reinterpret_cast<float*>(base + (ring - own));
    __nv_bfloat16* res = reinterpret_cast<__nv_bfloat16*>(sums + ROWS * LDF);
    if (far > 0) {
      far_stage<8>(sums, acc, rs, 0, lane);
      compute_sync<32 * CW>();
    }
    // the partial softmaxes of row r meet: weights 2^(m_k - m) / sum
    const float m0 = stat[r], m1 = stat[2 * ROWS + r], mf = far > 0 ? stat[4 * ROWS + r] : -INFINITY;
    const float mm = fmaxf(fmaxf(m0, m1), mf);               // finite: a query attends to itself
    float a0 = ex2(m0 - mm), a1 = ex2(m1 - mm), af = ex2(mf - mm);
    float total = fmaf(a0, stat[ROWS + r], a1 * stat[3 * ROWS + r]);
    if (far > 0) total = fmaf(af, stat[5 * ROWS + r], total);
    const float inv = 1.f / total;
    a0 *= inv;
    a1 *= inv;
    af *= inv;
    if (P.lse && half == 0 && ok) P.lse[((int64_t)b * P.heads + h) * P.seq + i] = (mm + log2f(total)) * 0.6931471805599453f;
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
      if (far > 0) {
#pragma unroll
        for (int e = 0; e < 16; e += 4) {
          const float4 y = *reinterpret_cast<const float4*>(sums + r * LDF + c + e);
          u[e] = __float_as_uint(fmaf(af, y.x, __uint_as_float(u[e])));
          u[e + 1] = __float_as_uint(fmaf(af, y.y, __uint_as_float(u[e + 1])));
          u[e + 2] = __float_as_uint(fmaf(af, y.z, __uint_as_float(u[e + 2])));
          u[e + 3] = __float_as_uint(fmaf(af, y.w, __uint_as_float(u[e + 3])));
        }
      }
      stage_row(res, r, c, u, nullptr, 1.f);
    }
    compute_sync<32 * CW>();
    if (ok) write_rows<16>(res, warp * 16, P.Out + h * D, (int64_t)row0 + q0, P.ldo, lane);
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
  CUtensorMap tmQ, tmK, tmV;
  if (!tile_map(&tmQ, Q, rows, width, ld) || !tile_map(&tmK, K, rows, width, ld) || !tile_map(&tmV, V, rows, width, ld)) return MST_ERR_SHAPE;
  FwdParams P;
  P.Out = (__nv_bfloat16*)Out;
  P.ldo = ldo;
  P.lse = lse;
  P.seq = seq_len; P.heads = heads;
  P.stride = stride < seq_len ? stride : seq_len;   // from there on the same pairs: all earlier positions
  P.magic = stride_magic(P.stride, seq_len);
  MST_SMEM_LIMIT((strided_attention_fwd_kernel), SMEM_BYTES);
  MST_CUDA_TRY(mst_launch_overlapped(strided_attention_fwd_kernel, dim3((unsigned)(seq_len / ROWS), (unsigned)heads, (unsigned)batch), dim3(THREADS),
                                     SMEM_BYTES, (cudaStream_t)stream, tmQ, tmK, tmV, P));
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}
