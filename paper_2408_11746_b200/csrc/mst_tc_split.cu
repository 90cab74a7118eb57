// fp32 contraction on the 5th-generation tensor cores: every fp32 operand is cut into three bf16 pieces whose sum is
// exactly the operand (8 + 8 + 8 significand bits; times 2^16, so that bf16's range holds the last bits of small values), and the product is the sum of the six piece products down to
// 2^-18 of the leading one.  The three products left out are below 2^-26 of |a b| together, less than the rounding of
// one fp32 multiplication.
//
// Sums.  The tensor core adds into an fp32 accumulator with truncation, so a long chain of additions would drift by
// more than an fp32 FMA chain does.  Therefore the leading products (a0 b0) and the five small ones go to accumulators
// of their own, and both are emptied into registers, with ordinary rounded fp32 additions, every 64 contraction
// indices: at most four truncating additions meet a sum of full size.  Error against fp64 (2-norm, normal operands):
// 0.7-0.9e-7 for the 3072 x 768 layer at 256 tokens, 1.0-1.6e-7 for 2048 x 4096 at 1024 tokens, where the FMA chains of the
// CUDA-core kernels leave 2.5-5e-7 and 6-12e-7 (emptied every 256 indices: 2.3e-7, all of it drift).
//
// What bounds it: six bf16 MMAs per fp32 product, so 1654 / 6 = 276 TFLOP/s of the measured bf16 peak against 74 for the
// fp32 FMA pipe; at the few hundred tokens of the fp32 workloads the launch, the pipeline fill and the drain of one tile
// cost as much as the products.  Hence small tiles (128 x 64) when the output has few of them, and a split of the
// contraction range over the blocks of a cluster, which add their sums through distributed shared memory in a fixed order
// (partial sums through global memory with the last block adding them cost 4 us more).  3072 x 768, d = 0.25, 256
// tokens: forward, input gradient and dense gradient with their operand preparation took 65 + 118 + 51 us on the CUDA
// cores (69 / 123 / 51 with their transposes), about 20 us each here.
//
// The same kernel with one piece serves bf16 contractions whose output has too few 256 x 256 tiles to occupy the GPU
// (mst_tc_small): small tiles and a split of the contraction range inside one launch.
//
// One block per tile and range, 320 threads: one lane of warp 0 fetches [3 pieces x rows x 64] boxes with TMA, one lane of
// warp 1 issues the MMAs, warps 2-9 own the sums (one row and BN / 2 columns per thread).  Every wait is bounded.
#include <cuda.h>

#include <atomic>

#include "mst_bits.cuh"
#include "mst_internal.cuh"
#include "mst_redo.cuh"
#include "mst_tc_gemm.cuh"
#include "mst_tc_ptx.cuh"

namespace {

using namespace mst_ptx;

__device__ int g_split_error = 0;  // sticky: a bounded wait expired

constexpr int SBM = 128, SBK = 64;
constexpr int S_EPI_WARPS = 8;
constexpr int S_THREADS = 64 + 32 * S_EPI_WARPS;
constexpr int BOX64 = 64 * SBK * 2;         // one piece of one 64-wide MN-major box

template <int BN, int PIECES>
struct SplitCfg {
  static constexpr int CHUNK_KB = PIECES == 3 ? 1 : 1 << 20;   // k-blocks summed inside the tensor core before the sums move to registers
  static constexpr int A_BYTES = PIECES * SBM * SBK * 2;
  static constexpr int B_BYTES = PIECES * BN * SBK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  // one piece: at most half of an SM's shared memory, so that the next launch's blocks can be set up while this one drains
  static constexpr int STAGES = PIECES == 1 ? 4 : BN == 64 ? 3 : 2;
  static constexpr int TMEM = PIECES == 3 ? 4 * BN : BN;       // three pieces: two chunk buffers x (leading, small)
  // after the last MMA the stages hold the warps' turning squares and the block's sums
  static constexpr int STAGING = S_EPI_WARPS * 32 * 33 * 4 + SBM * BN * 4;
  static constexpr int TILES = STAGES * STAGE_BYTES > STAGING ? STAGES * STAGE_BYTES : STAGING;
  static constexpr size_t SMEM = (size_t)TILES + 1024 /*align*/ + 128 /*barriers*/;
};

struct SplitParams {
  int64_t M, N;
  int kblocks, splits, m_tiles, n_tiles;
  void* out;
  uint16_t* pre;
  int64_t ldpre;
  int64_t ldc;
  const uint32_t* bits;
  const int32_t* wscan;
  int wpr;
  float* entries;   // S_BOTH
  int kind, major;
  mst_redo redo;
};

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, int x, int y, int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(tm), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}

// all warps of all blocks of the cluster, converged
__device__ __forceinline__ void split_cluster_sync() {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Sums of a 32-column square over the 2^LG blocks of the cluster, this block's 32 / 2^LG rows from rr0 on, into the warp's box: a
// lane adds four columns of some rows, eight reads whatever the number of blocks, all in flight together, added in range order.
// Returns 0 if this lane's sums are finite, else NaN.
template <int LG, int PIECES>
__device__ __forceinline__ float gather_sums(uint32_t sums, int rr0, float* box, int lane) {
  float4 x[8];
  float zero = 0.f;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int i = lane + 32 * (j >> LG), row = rr0 + (i >> 3);
    uint32_t peer;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(peer) : "r"(sums + (uint32_t)((i & 7) * 32 + row) * 16u), "r"(j & ((1 << LG) - 1)));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(x[j].x), "=f"(x[j].y), "=f"(x[j].z), "=f"(x[j].w) : "r"(peer) : "memory");
  }
#pragma unroll
  for (int j = 0; j < 8; j += 1 << LG) {
    float4 sum = x[j];
#pragma unroll
    for (int k = 1; k < 1 << LG; ++k) { sum.x += x[j + k].x; sum.y += x[j + k].y; sum.z += x[j + k].z; sum.w += x[j + k].w; }
    if (PIECES == 3) { sum.x *= MST_SPLIT_UNSCALE; sum.y *= MST_SPLIT_UNSCALE; sum.z *= MST_SPLIT_UNSCALE; sum.w *= MST_SPLIT_UNSCALE; }
    const int i = lane + 32 * (j >> LG);
    float* d = box + (rr0 + (i >> 3)) * 33 + 4 * (i & 7);
    d[0] = sum.x; d[1] = sum.y; d[2] = sum.z; d[3] = sum.w;
    zero = fmaf(sum.x, 0.f, fmaf(sum.y, 0.f, fmaf(sum.z, 0.f, fmaf(sum.w, 0.f, zero))));
  }
  return zero;
}

// Rows rr0 .. end - 1 of this lane's column of the warp's box, four at a time: read back together, then handed on one by one.  Nothing
// is tested per store - a test, with its branch and its 64-bit address, made 64 KB of stores take 8000 clocks instead of 2200, and
// the last token tile of 600 tokens, whose rows went one by one, cost each call 1.6 us.
template <typename Store>
__device__ __forceinline__ void box_rows(const float* box, int rr0, int end, int lane, Store store) {
  int r = rr0;
#pragma unroll 2
  for (; r + 4 <= end; r += 4) {
    float v[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) v[k] = box[(r + k) * 33 + lane];
#pragma unroll
    for (int k = 0; k < 4; ++k) store(r + k, v[k]);
  }
#pragma unroll 1
  for (; r < end; ++r) store(r, box[r * 33 + lane]);
}

// One kernel for every kind of output and the operands' majors, but for the activations.  A kernel each takes 0.3 to 0.5 us less where one call
// repeats (3072 x 768 in fp32, 256 tokens: 17.8 against 18.2), but a pass takes turns, and each then fetches its instructions anew: the three
// products of small layers, a kernel each / one, fp32 495 x 96 at 208 tokens 29.8 / 27.7 us, 320 x 576 at 75 31.2 / 29.7, 1114 x 256 at 253 38.5 / 37.0,
// bf16 896 x 111 at 925 28.7 / 26.9, 256 x 383 at 785 26.7 / 24.7; 2.4 % over thirty fp32 layers of 96..2048 features, 0.7 % over thirty in bf16.
enum {
  S_F32, S_SAMPLED,
  S_BOTH,   // fp32, and its entries under the mask
  S_BF16
};
enum { M_FORWARD, M_INPUT, M_GRADIENT };   // MN-major operands: none, the second, both

template <int BN, int PIECES, int ACT>
__global__ void __launch_bounds__(S_THREADS, PIECES == 1 ? 2 : 1)
tc_split_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB, const SplitParams P) {
  typedef SplitCfg<BN, PIECES> C;
  constexpr int CHUNK_KB = C::CHUNK_KB;
  const int kind = ACT ? S_BF16 : P.kind;
  const bool a_mn = !ACT && P.major == M_GRADIENT, b_mn = ACT ? ACT == MST_ACT_GELU_GRAD : P.major != M_FORWARD;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles_base = (raw + 1023u) & ~1023u;
  const uint32_t bar_base = tiles_base + C::TILES;
  const uint32_t full0 = bar_base, empty0 = full0 + 8 * C::STAGES, tfull0 = empty0 + 8 * C::STAGES, tempty0 = tfull0 + 16;
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < C::STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, S_EPI_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmA) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(&tmB) : "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)), "r"(C::TMEM)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  const int split = P.splits > 1 ? (int)(blockIdx.x % (unsigned)P.splits) : 0, tile = (int)(blockIdx.x / (unsigned)P.splits);   // rank in the cluster
  const int m0 = (tile / P.n_tiles) * SBM, n0 = (tile % P.n_tiles) * BN;
  const int kb0 = (int)((int64_t)split * P.kblocks / P.splits), kb1 = (int)((int64_t)(split + 1) * P.kblocks / P.splits);
  const int chunks = (kb1 - kb0 + CHUNK_KB - 1) / CHUNK_KB;

  if (warp == 0) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      for (int kb = kb0; kb < kb1; ++kb) {
        if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag, &g_split_error)) break;
        const uint32_t fb = full0 + 8 * s, sa = tiles_base + s * C::STAGE_BYTES, sb = sa + C::A_BYTES;
        mbar_expect_tx(fb, C::STAGE_BYTES);
        if (a_mn) {
          for (int j = 0; j < SBM / 64; ++j) tma_load_3d(sa + j * PIECES * BOX64, &tmA, m0 + j * 64, kb * SBK, 0, fb);
        } else {
          tma_load_3d(sa, &tmA, kb * SBK, m0, 0, fb);
        }
        if (b_mn) {
          for (int j = 0; j < BN / 64; ++j) tma_load_3d(sb + j * PIECES * BOX64, &tmB, n0 + j * 64, kb * SBK, 0, fb);
        } else {
          tma_load_3d(sb, &tmB, kb * SBK, n0, 0, fb);
        }
        if (++s == C::STAGES) { s = 0; ph ^= 1u; }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(a_mn ? 1 : 0) << 15) |
                             ((uint32_t)(b_mn ? 1 : 0) << 16) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(SBM >> 4) << 24);
      // K-major: the three pieces of a stage lie one after the other; MN-major: 64-wide blocks, each with its three pieces
      const uint64_t ad0 = smem_desc(tiles_base, a_mn ? PIECES * BOX64 : 16, 1024);
      const uint64_t bd0 = smem_desc(tiles_base + C::A_BYTES, b_mn ? PIECES * BOX64 : 16, 1024);
      const uint32_t a_piece = (uint32_t)(a_mn ? BOX64 : SBM * SBK * 2) >> 4, b_piece = (uint32_t)(b_mn ? BOX64 : BN * SBK * 2) >> 4;
      const uint32_t a_k = (uint32_t)(a_mn ? 16 * 128 : 32) >> 4, b_k = (uint32_t)(b_mn ? 16 * 128 : 32) >> 4;
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int c = 0; c < chunks && ok; ++c) {
        const int buf = c & 1;
        if (!mbar_wait(tempty0 + 8 * buf, ((c >> 1) & 1) ^ 1u, abort_flag, &g_split_error)) break;
        tc_fence_after();
        const uint32_t d_hi = tmem_base + (uint32_t)(buf * 2 * BN), d_lo = d_hi + BN;
        const int first = kb0 + c * CHUNK_KB, last = first + CHUNK_KB < kb1 ? first + CHUNK_KB : kb1;
        for (int kb = first; kb < last; ++kb) {
          if (!mbar_wait(full0 + 8 * s, ph, abort_flag, &g_split_error)) { ok = false; break; }
          tc_fence_after();
          const uint64_t ad = ad0 + (uint64_t)(uint32_t)(s * (C::STAGE_BYTES >> 4)), bd = bd0 + (uint64_t)(uint32_t)(s * (C::STAGE_BYTES >> 4));
#pragma unroll
          for (int k = 0; k < SBK / 16; ++k) {
            const uint32_t more = (kb > first || k > 0) ? 1u : 0u;
            const uint64_t a0 = ad + (uint64_t)(k * a_k), b0 = bd + (uint64_t)(k * b_k);
            if (PIECES == 1) {
              tc_mma(d_hi, a0, b0, idesc, more);
              continue;
            }
            const uint64_t a1 = a0 + a_piece, a2 = a1 + a_piece, b1 = b0 + b_piece, b2 = b1 + b_piece;
            tc_mma(d_lo, a2, b0, idesc, more);
            tc_mma(d_lo, a0, b2, idesc, 1u);
            tc_mma(d_lo, a1, b1, idesc, 1u);
            tc_mma(d_lo, a1, b0, idesc, 1u);
            tc_mma(d_lo, a0, b1, idesc, 1u);
            tc_mma(d_hi, a0, b0, idesc, more);
          }
          tc_commit(empty0 + 8 * s);
          if (++s == C::STAGES) { s = 0; ph ^= 1u; }
        }
        if (ok) tc_commit(tfull0 + 8 * buf);
      }
    }
  } else {
    const int q = warp & 3, half = (warp - 2) >> 2;
    constexpr int COLS = BN / 2;   // columns of this thread's row
    float acc[COLS];
#pragma unroll
    for (int j = 0; j < COLS; ++j) acc[j] = 0.f;
    for (int c = 0; c < chunks; ++c) {
      const int buf = c & 1;
      if (!mbar_wait(tfull0 + 8 * buf, (c >> 1) & 1, abort_flag, &g_split_error)) break;
      tc_fence_after();
      const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(buf * 2 * BN + half * COLS);
#pragma unroll
      for (int g = 0; g < COLS / 32; ++g) {
        uint32_t hi[32], lo[32];
        tmem_ld32_nowait(at + g * 32, hi);
        if (PIECES == 3) tmem_ld32_nowait(at + BN + g * 32, lo);
        tmem_ld_wait(hi);
        if (PIECES == 3) tmem_ld_wait(lo);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[g * 32 + j] += PIECES == 3 ? __uint_as_float(hi[j]) + __uint_as_float(lo[j]) : __uint_as_float(hi[j]);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * buf);
    }
    // Every MMA of the block has completed, so the operand stages serve as staging.
    float* box = reinterpret_cast<float*>(smem_raw + (tiles_base - raw)) + (warp - 2) * (32 * 33);
    const uint32_t part = tiles_base + S_EPI_WARPS * 32 * 33 * 4 + (uint32_t)((warp - 2) * (COLS / 4) * 32 + lane) * 16u;
    int rr0 = 0, rr1 = 32;   // rows of the warp's 32 this block stores
    if (P.splits > 1) {
      // The blocks of a cluster hold the sums of one tile over different parts of the contraction range: each leaves its sums in
      // its shared memory, then adds up and stores 32 / splits of every 32 rows, in range order.
#pragma unroll
      for (int v = 0; v < COLS / 4; ++v)
        asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(part + v * 512u), "f"(acc[4 * v]), "f"(acc[4 * v + 1]), "f"(acc[4 * v + 2]),
                     "f"(acc[4 * v + 3])
                     : "memory");
      split_cluster_sync();
      rr0 = split * (32 / P.splits);
      rr1 = rr0 + 32 / P.splits;
    }
    if (!*abort_flag) {
      // a 32 x 32 square per warp, turned from rows to columns so that a store instruction writes neighbours
      const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
      for (int g = 0; g < COLS / 32; ++g) {
        const int n = n0 + half * COLS + g * 32;
        if (n >= P.N) break;   // uniform
        __syncwarp();
        float zero = 0.f;   // NaN where a sum is not finite
        if (P.splits > 1) {
          if (P.splits == 2) zero = gather_sums<1, PIECES>(part - (uint32_t)lane * 16u + (uint32_t)(g * 8 * 32) * 16u, rr0, box, lane);
          else if (P.splits == 4) zero = gather_sums<2, PIECES>(part - (uint32_t)lane * 16u + (uint32_t)(g * 8 * 32) * 16u, rr0, box, lane);
          else zero = gather_sums<3, PIECES>(part - (uint32_t)lane * 16u + (uint32_t)(g * 8 * 32) * 16u, rr0, box, lane);
        } else {
#pragma unroll
          for (int j = 0; j < 32; ++j) zero = fmaf(acc[g * 32 + j], 0.f, zero);
#pragma unroll
          for (int j = 0; j < 32; ++j) box[lane * 33 + j] = PIECES == 3 ? acc[g * 32 + j] * MST_SPLIT_UNSCALE : acc[g * 32 + j];
        }
        __syncwarp();
        const int64_t row0 = (int64_t)m0 + q * 32;
        if (P.redo.kind && __any_sync(0xffffffffu, zero != 0.f)) {
          const bool mine = lane >= rr0 && lane < rr1 && row0 + lane < P.M;
          if (PIECES == 3) mst_redo_square<float>(P.redo, box + lane * 33, row0 + lane, mine, n, P.N);
          else mst_redo_square<uint16_t>(P.redo, box + lane * 33, row0 + lane, mine, n, P.N);
          __syncwarp();
        }
        const int end = n + lane >= P.N ? 0 : (int)(P.M - row0 < rr1 ? P.M - row0 : rr1);   // rows of this lane's column
        if (kind == S_SAMPLED || kind == S_BOTH) {
          uint32_t word = 0;
          int32_t at = 0;
          if (row0 + lane < P.M) {
            const int64_t wi = (row0 + lane) * P.wpr + (n >> 5);
            word = P.bits[wi];
            at = P.wscan[wi];
          }
          float* out = kind == S_BOTH ? P.entries : reinterpret_cast<float*>(P.out);
          box_rows(box, rr0, rr1, lane, [&](int rr, float v) {   // words beyond the matrix are empty
            const uint32_t w = __shfl_sync(0xffffffffu, word, rr);
            const int32_t base = __shfl_sync(0xffffffffu, at, rr);
            if ((w >> lane) & 1u) out[base + __popc(w & lt)] = v;
          });
        }
        if (PIECES == 1 && kind == S_BF16) {
          uint16_t* out = reinterpret_cast<uint16_t*>(P.out) + row0 * P.ldc + n + lane;
          uint16_t* pre = P.pre + row0 * P.ldpre + n + lane;
          if (ACT == MST_ACT_NONE)
            box_rows(box, rr0, end, lane,
                     [&](int rr, float v) { out[rr * P.ldc] = (uint16_t)(pack_bf16(v, 0.f) & 0xFFFFu); });
          else if (ACT == MST_ACT_GELU_GRAD) {   // the derivative at the stored pre-activation
            // sixteen rows' inputs at a time, before any of their results leaves: row by row each waits out its load (64 tokens,
            // 192 x 768: 11.6 us).  Rows past the end repeat the last one, so that only the stores are conditional and the sixteen
            // derivatives overlap.
#pragma unroll 1
            for (int r = rr0; r < end; r += 16) {
              uint16_t x[16];
              float y[16];
#pragma unroll
              for (int k = 0; k < 16; ++k) x[k] = pre[(r + k < end ? r + k : end - 1) * P.ldpre];
#pragma unroll
              for (int k = 0; k < 16; ++k)
                y[k] = box[(r + k < end ? r + k : end - 1) * 33 + lane] * mst_gelu_grad(__uint_as_float((uint32_t)x[k] << 16));
#pragma unroll
              for (int k = 0; k < 16; ++k)
                if (r + k < end) out[(r + k) * P.ldc] = (uint16_t)(pack_bf16(y[k], 0.f) & 0xFFFFu);
            }
          } else
            box_rows(box, rr0, end, lane, [&](int rr, float v) {
              if (P.pre) pre[rr * P.ldpre] = (uint16_t)(pack_bf16(v, 0.f) & 0xFFFFu);
              out[rr * P.ldc] = (uint16_t)(pack_bf16(mst_gelu(v), 0.f) & 0xFFFFu);
            });
        } else if (kind != S_SAMPLED) {
          float* out = reinterpret_cast<float*>(P.out) + row0 * P.ldc + n + lane;
          box_rows(box, rr0, end, lane, [&](int rr, float v) { out[rr * P.ldc] = v; });
        }
      }
    }
  }

  if (P.splits > 1) {
    if (warp < 2) split_cluster_sync();   // the barrier above, for the warps without sums
    split_cluster_sync();                 // no block leaves while another still reads its sums
  }
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);  // copies and MMAs in flight land before memory is given back
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(C::TMEM) : "memory");
  }
}

// pieces [1 or 3][rows][ld] as a 3-d map: rows and columns beyond the matrix read as zero inside every piece
bool make_piece_map(CUtensorMap* tm, const void* base, int pieces, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn) return false;
  cuuint64_t dims[3] = {(cuuint64_t)cols, (cuuint64_t)rows, (cuuint64_t)pieces};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 2, (cuuint64_t)(ld * rows) * 2};
  cuuint32_t box[3] = {64u, (cuuint32_t)box_rows, (cuuint32_t)pieces};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int BN, int PIECES, int ACT>
mst_status_t launch_split(const CUtensorMap& tmA, const CUtensorMap& tmB, const SplitParams& P, cudaStream_t s) {
  typedef SplitCfg<BN, PIECES> C;
  MST_SMEM_LIMIT((tc_split_kernel<BN, PIECES, ACT>), C::SMEM);
  MST_CUDA_TRY(mst_launch_overlapped_cluster(tc_split_kernel<BN, PIECES, ACT>, dim3((unsigned)(P.m_tiles * P.n_tiles * P.splits)),
                                             dim3(S_THREADS), P.splits, C::SMEM, s, tmA, tmB, P));
  return MST_OK;
}
// Blocks that run at once, one to an SM, in clusters of 1 .. 8: the groups of SMs that a cluster must fit into are no multiples of it (148
// SMs hold 148, 148, 132 and 120 blocks in clusters of 1, 2, 4 and 8).  Asked once per device, and for the device once a plan: asked for every width and
// number of ranges the plans of a forward call cost it 0.5 us.
struct Slots { int in[9]; };
Slots cluster_slots() {
  static std::atomic<int> known[64][9];
  Slots found;
  int dev = 0;
  const bool here = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < 64;
  int sms = here ? known[dev][1].load(std::memory_order_relaxed) : 0;
  if (sms == 0) sms = mst_sm_count();
  for (int& n : found.in) n = sms;
  if (!here) return found;
  known[dev][1].store(sms, std::memory_order_relaxed);
  for (int size = 2; size <= 8; size *= 2) {
    int n = known[dev][size].load(std::memory_order_relaxed);
    if (n == 0) {
      typedef SplitCfg<128, 3> C;   // one block to an SM
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3((unsigned)(size * sms));
      cfg.blockDim = dim3(S_THREADS);
      cfg.dynamicSmemBytes = C::SMEM;
      cudaLaunchAttribute attr;
      attr.id = cudaLaunchAttributeClusterDimension;
      attr.val.clusterDim.x = (unsigned)size;
      attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
      cfg.attrs = &attr;
      cfg.numAttrs = 1;
      int clusters = 0;
      if (cudaFuncSetAttribute(tc_split_kernel<128, 3, MST_ACT_NONE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)C::SMEM) != cudaSuccess ||
          cudaOccupancyMaxActiveClusters(&clusters, tc_split_kernel<128, 3, MST_ACT_NONE>, &cfg) != cudaSuccess || clusters <= 0) {
        cudaGetLastError();   // reported by the launch, if it matters there
        continue;
      }
      n = clusters * size < sms ? clusters * size : sms;
      known[dev][size].store(n, std::memory_order_relaxed);
    }
    found.in[size] = n;
  }
  return found;
}

// Tile width and number of K ranges from a time model in SM clocks.
// Three pieces: 24 MMAs per k-block (64 clocks each at 128 columns, 40 at 64, where the A operand's shared-memory reads dominate),
// about 10000 for launch, fill and drain of a wave, and 1500 for the sums of a cluster.
// One piece (64 columns; 128 were no faster), at 1.85 GHz: a launch, the k-blocks (24 KB of operands each), a further wave, the sums of
// a cluster; two blocks share an SM, in clusters as well, each then a little slower.
// All choices timed for 138 fp32 and 190 bf16 layers drawn over 96..4096 x 96..2048 features and the widths of a block up to 1280, 64..1024
// (fp32) and 17..4096 tokens; 138 and 189 further ones for the check.  With 148 blocks assumed at any cluster size and one of a cluster to
// an SM, ranges over eight blocks were taken where two or four are faster: fp32 calls 4.5 % above the best choice of each, now 0.6;
// the further ones take 0.965 of that time, bf16 products of few tiles 0.96 (1024 x 1024 at 162 tokens, fp32: 21.9 -> 13.7 us; bf16 input
// gradient 4352 -> 1088 at 710 tokens 21.8 -> 16.8).  Gradients of one piece: see mst_tc_choose.
mst_small_plan plan_split(const mst_tc_gemm_args& a, int pieces) {
  struct Figures { double launch, wave, k_shared, shared, cluster; };
  static const Figures plain = {7160.0, 0.0, 483.0, 1490.0, 5940.0}, gelu = {10700.0, 1550.0, 515.0, 1640.0, 2440.0},
                       grad = {13000.0, 2500.0, 512.0, 1980.0, 1700.0},
                       sampled = {9070.0, 0.0, 496.0, 1620.0, 3690.0}, f32 = {9290.0, 0.0, 450.0, 850.0, 3510.0}, both = {9670.0, 0.0, 481.0, 2680.0, 3460.0};
  const Slots slots = cluster_slots();
  const int sms = slots.in[1], kblocks = (int)((a.K + SBK - 1) / SBK);
  const int64_t m_tiles = (a.M + SBM - 1) / SBM;
  const bool gradient = a.epilogue != MST_TC_OUT_BF16, even = a.M % 8 == 0 && a.N % 8 == 0;
  mst_small_plan best = {64, 1, 1e30};
  for (int w = 64; w <= (pieces == 3 ? 128 : 64); w += 64) {
    const int64_t tiles = m_tiles * ((a.N + w - 1) / w);
    for (int sp = 1; sp <= 8 && sp <= kblocks; sp *= 2) {   // cluster sizes
      const int kb = (kblocks + sp - 1) / sp, fit = slots.in[sp];
      double t;
      if (pieces == 3) {
        const int64_t waves = (tiles * sp + fit - 1) / fit;
        t = (double)waves * (kb * (w == 64 ? 960.0 : 1620.0) + 10000.0) + (sp > 1 ? 1500.0 : 0.0);
      } else if (!gradient || even) {
        const Figures& F = a.epilogue == MST_TC_OUT_SAMPLED ? sampled : gradient ? (a.also_sampled ? both : f32) : a.act == MST_ACT_GELU_GRAD ? grad : a.act ? gelu : plain;
        const int64_t waves = (tiles * sp + 2 * fit - 1) / (2 * fit);
        const double pair = kb * F.k_shared, alone = kb * (!gradient ? 471.0 : a.epilogue == MST_TC_OUT_SAMPLED ? 432.0 : a.also_sampled ? 478.0 : 389.0);
        t = F.launch + F.wave * (double)waves + (double)(waves - 1) * (11500.0 + pair) + (tiles * sp > fit ? pair + F.shared : alone) + (sp > 1 ? F.cluster : 0.0);
      } else {
        // gradients of odd sizes: copies ahead, partial squares.  Entries are nearer to the best with one block of a cluster to an SM (1.4 % above it
        // against 1.7), dense ones with two (1.1 against 1.5).
        const int64_t most = a.epilogue != MST_TC_OUT_SAMPLED || sp == 1 ? 2 * fit : sms, waves = (tiles * sp + most - 1) / most;
        t = 9000.0 + (double)waves * kb * 555.0 + (double)(waves - 1) * 10000.0 + (sp > 1 ? 5000.0 : 0.0);
      }
      if (t < best.clocks * 0.97) best = {w, sp, t};
    }
  }
  return best;
}

mst_status_t run_split(const mst_tc_gemm_args& a, int pieces, int bn, int splits, cudaStream_t s) {
  SplitParams P = {};
  P.M = a.M;
  P.N = a.N;
  P.kblocks = (int)((a.K + SBK - 1) / SBK);
  P.m_tiles = (int)((a.M + SBM - 1) / SBM);
  P.n_tiles = (int)((a.N + bn - 1) / bn);
  P.splits = splits;
  P.out = a.out;
  P.ldc = a.ldc;
  P.pre = (uint16_t*)a.pre;
  P.ldpre = a.ldpre;
  P.bits = a.bits;
  P.wscan = a.wscan;
  P.wpr = a.wpr;
  P.redo = a.redo;
  // The squares are in shared memory already; a sweep over the finished matrix for its entries costs a launch and reads it again.
  // Dense gradient with its entries: fp32 3072 x 768, 256 tokens 20.9 -> 18.6 us; bf16 1216 x 1216, 534 tokens 11.1 -> 8.9.
  if (a.epilogue == MST_TC_OUT_F32 && a.also_sampled) {
    P.entries = a.also_sampled;
    *a.sampled = true;
  }
  const int act = a.epilogue == MST_TC_OUT_BF16 ? a.act : 0, major = a.a_mn_major ? M_GRADIENT : a.b_mn_major ? M_INPUT : M_FORWARD;
  if (act == MST_ACT_GELU_GRAD && !P.pre) return MST_ERR_INVALID_ARG;
  // the forms that the entry points have: GELU forward and its derivative backward; one piece: products in bf16, gradients in fp32
  if (act && (act == MST_ACT_GELU_GRAD) != (major == M_INPUT)) return MST_ERR_INVALID_ARG;
  if (pieces == 1 && (a.epilogue == MST_TC_OUT_BF16) == (major == M_GRADIENT)) return MST_ERR_INVALID_ARG;
  if (a.epilogue == MST_TC_OUT_SAMPLED && major != M_GRADIENT) return MST_ERR_INVALID_ARG;
  CUtensorMap tmA, tmB;
  const bool okA = a.a_mn_major ? make_piece_map(&tmA, a.A, pieces, a.K, a.M, a.lda, SBK) : make_piece_map(&tmA, a.A, pieces, a.M, a.K, a.lda, SBM);
  const bool okB = a.b_mn_major ? make_piece_map(&tmB, a.B, pieces, a.K, a.N, a.ldb, SBK) : make_piece_map(&tmB, a.B, pieces, a.N, a.K, a.ldb, bn);
  if (!okA || !okB) return MST_ERR_SHAPE;
  P.major = major;
  P.kind = a.epilogue == MST_TC_OUT_SAMPLED ? S_SAMPLED : a.epilogue == MST_TC_OUT_BF16 ? S_BF16 : P.entries ? S_BOTH : S_F32;
  if (pieces == 3) return bn == 64 ? launch_split<64, 3, MST_ACT_NONE>(tmA, tmB, P, s) : launch_split<128, 3, MST_ACT_NONE>(tmA, tmB, P, s);
  return act == MST_ACT_GELU ? launch_split<64, 1, MST_ACT_GELU>(tmA, tmB, P, s)
         : act ? launch_split<64, 1, MST_ACT_GELU_GRAD>(tmA, tmB, P, s) : launch_split<64, 1, MST_ACT_NONE>(tmA, tmB, P, s);
}

}  // namespace

mst_status_t mst_tc_split(const mst_tc_gemm_args& a, cudaStream_t s) {
  const mst_small_plan plan = plan_split(a, 3);
  return run_split(a, 3, plan.bn, plan.splits, s);
}

mst_small_plan mst_tc_small_plan(const mst_tc_gemm_args& a) { return plan_split(a, 1); }

mst_status_t mst_tc_small(const mst_tc_gemm_args& a, const mst_small_plan& plan, cudaStream_t s) { return run_split(a, 1, plan.bn, plan.splits, s); }

mst_status_t mst_split_error_flags(int32_t* flags) {
  int v = 0;
  MST_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_split_error, sizeof(int)));
  *flags = v;
  return MST_OK;
}
