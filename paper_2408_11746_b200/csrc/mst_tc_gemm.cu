// bf16 contraction on the 5th-generation tensor cores (tcgen05) with fp32 accumulators in tensor memory.
//
// One persistent block per SM, 320 threads in three roles:
//   warp 0     producer: one lane issues TMA tile loads (cp.async.bulk.tensor, 128-byte swizzle) into a 4-stage
//              shared-memory ring, signalling "full" mbarriers by transaction bytes;
//   warp 1     one lane issues tcgen05.mma (M=128, N=256, K=16 per instruction) from shared-memory descriptors
//              into one of two 128x256 fp32 accumulators in tensor memory, tcgen05.commit releases the smem stage
//              ("empty") and, after the last K block, hands the accumulator to the epilogue ("tmem_full");
//   warps 2-9  epilogue, two warps per tensor-memory lane quarter taking alternate 32-column chunks: tcgen05.ld
//              (one row per thread), convert / activate / sample / store, then release the accumulator
//              ("tmem_empty") so the next tile's MMAs overlap this tile's stores.
// Operands may be K-major ([rows x K] row-major) or MN-major ([K x rows] row-major, as dY and X are for
// G = dY^T X): the tile is fetched with 64-element-wide boxes either way and described to the tensor core with the
// matching canonical layout (K-major: 8-row groups 1024 B apart; MN-major: 64-wide blocks one box apart).
// Every mbarrier wait is bounded: on expiry the block raises an abort flag, records an error bit, skips the rest
// of its work, frees its tensor memory and returns.
#include "mst_tc_gemm.cuh"

#include <cuda.h>
#include <cuda_bf16.h>

#include <cstdlib>

#include "mst_internal.cuh"
#include "mst_redo.cuh"
#include "mst_tc_ptx.cuh"

namespace {

constexpr int BM = 128, BN = 256, BK = 64, STAGES = 4, UMMA_K = 16;
constexpr int A_BYTES = BM * BK * 2;  // 16 KiB
constexpr int B_BYTES = BN * BK * 2;  // 32 KiB
constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
constexpr int BOX_BYTES = 64 * BK * 2;  // one 64-wide MN-major box: 8 KiB
constexpr int EPI_WARPS = 8;  // two per tensor-memory lane quarter, alternating 32-column chunks
constexpr int NUM_THREADS = 64 + 32 * EPI_WARPS;
constexpr int TMEM_COLS = 512;
constexpr int OUT_BOX_BYTES = 32 * 128;  // one epilogue warp's staging box: 32 rows x 128 bytes
constexpr size_t SMEM_BYTES = (size_t)STAGES * STAGE_BYTES + EPI_WARPS * OUT_BOX_BYTES + 1024 /*align*/ + 256 /*barriers*/;

__device__ int g_tc_error = 0;  // sticky: 1 = a bounded wait expired

struct Params {
  int64_t M, N;
  int kblocks;        // ceil(K / BK)
  int splits;
  int m_tiles, n_tiles;
  uint32_t full, cut; // pair kernel: whole jobs, and how many each later one is cut into (rows: two halves; gradients: K ranges)
  int epilogue;
  int major;
  void* out;
  int64_t ldc;
  float* partial;
  const uint32_t* bits;
  const int32_t* wscan;
  int wpr;
  int64_t nnz;
  int act;
  void* pre;
  int64_t ldpre;
  int whole;    // bf16 rows by TMA: columns up to here, the last whole 16 bytes of a row, are in the map; the others leave by the lanes
  mst_redo redo;          // rows of bf16: sums that are not finite are formed again
  int sampled_stage_min;  // sampled output: a 32 x 32 chunk with at least this many kept entries leaves row by row
};

// How the accumulators leave: a kernel each, and the operands' majors are constants of the pair kernel too.  What a launch does not
// run costs it all the same: with one kernel for everything (168 registers where rows of bf16 alone need 62, and cold branches
// between the hot ones) each product paid 0.4 us a launch and 20 clocks a k-block for it.  8192 tokens, forward / input gradient:
// 768 x 768 13.3 / 13.2 -> 11.6 / 11.5 us, 3072 x 768 32.4 / 36.4 -> 29.7 / 32.5, 768 x 3072 36.5 / 32.2 -> 32.3 / 29.7; entries under
// the mask 17.9 -> 16.1, 32.8 -> 32.0, 34.2 -> 32.6.  A training pass that alternates between them gains as much.
// Which operands are MN-major: none (activations x image), the second (gradients x image), both (gradients x activations)
enum { M_FORWARD, M_INPUT, M_GRADIENT };
enum {
  K_BF16, K_F32, K_SAMPLED,
  K_ACT,    // bf16 with an activation
  // bf16 without and with one, where sums that are not finite are formed again or rows end inside a 16-byte piece.  (One kernel for both, a ring
  // stage short: 770 -> 3072 at 8192 tokens 38.3 -> 37.3 us, its input gradient 37.1 -> 36.3.  The ends of rows seen to in the kernels above: 1 to 2 %
  // of theirs.)
  K_REDO, K_REDO_ACT,
  K_ROWS, K_ROWS_ACT    // whatever the TMA unit cannot describe, without and with an activation
};

// PTX wrappers live in mst_tc_ptx.cuh; waits in this file report to g_tc_error
using namespace mst_ptx;
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag) {
  return mst_ptx::mbar_wait(bar, parity, abort_flag, &g_tc_error);
}

// Phi(x) and exp(-x^2/2) for the fused activation.  The complementary error function is the five-term rational
// approximation of Abramowitz & Stegun 7.1.26 (absolute error below 1.5e-7, far under the bf16 rounding of the
// result); it shares its exponential with the normal density, and Phi of a negative argument is formed without
// cancellation.  It costs about a third of erff's instructions (flush-to-zero reciprocal and exp2, whose default
// forms carry denormal handling); the epilogue is still the slower side of the overlap when an activation is fused.
__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Two values at a time: the fp32 pipe takes a register pair per instruction, which halves the issue slots of everything but the
// reciprocals and exponentials (10 a value against 17; times at epilogue_tile_act).
// -Phi(-|x|) and exp(-x^2 / 2) of a pair; the five coefficients carry the factor -1/2
__device__ __forceinline__ void phi_pair(float x0, float x1, uint64_t& nq, uint64_t& e) {
  const uint64_t t_arg = fma2(pack2(fabsf(x0), fabsf(x1)), pack2(0.3275911f * 0.70710678118654752f, 0.3275911f * 0.70710678118654752f), pack2(1.0f, 1.0f));
  float t0, t1, y0, y1;
  unpack2(t_arg, t0, t1);
  const uint64_t t = pack2(rcp_approx(t0), rcp_approx(t1)), x = pack2(x0, x1);
  unpack2(mul2(mul2(x, x), pack2(-0.72134752044448170f, -0.72134752044448170f)), y0, y1);
  e = pack2(ex2_approx(y0), ex2_approx(y1));   // exp(-x^2 / 2)
  uint64_t poly = fma2(t, pack2(-0.5f * 1.061405429f, -0.5f * 1.061405429f), pack2(0.5f * 1.453152027f, 0.5f * 1.453152027f));
  poly = fma2(poly, t, pack2(-0.5f * 1.421413741f, -0.5f * 1.421413741f));
  poly = fma2(poly, t, pack2(0.5f * 0.284496736f, 0.5f * 0.284496736f));
  poly = fma2(poly, t, pack2(-0.5f * 0.254829592f, -0.5f * 0.254829592f));
  nq = mul2(mul2(poly, t), e);
}
// x Phi(x) = max(x, 0) - |x| Phi(-|x|).  The factor of the vanishing term stays finite for x = +inf (the result is +inf); -inf gives
// NaN, as the product x Phi(x) does.
__device__ __forceinline__ void gelu_pair(float& x0, float& x1) {
  uint64_t nq, e;
  phi_pair(x0, x1, nq, e);
  const uint64_t ax = pack2(fabsf(fminf(x0, 3.4028235e38f)), fabsf(fminf(x1, 3.4028235e38f)));
  unpack2(fma2(ax, nq, pack2(fmaxf(x0, 0.f), fmaxf(x1, 0.f))), x0, x1);
}
// d/dx x Phi(x) = Phi(x) + x phi(x): with u = |x| phi(x) - Phi(-|x|) it is 1 + u right of zero and -u left of it (by the sign bit)
__device__ __forceinline__ uint64_t gelu_grad_pair(float x0, float x1) {
  uint64_t nq, e;
  phi_pair(x0, x1, nq, e);
  float u0, u1;
  unpack2(fma2(mul2(pack2(fabsf(x0), fabsf(x1)), pack2(0.39894228040143268f, 0.39894228040143268f)), e, nq), u0, u1);
  const uint32_t s0 = __float_as_uint(x0) & 0x80000000u, s1 = __float_as_uint(x1) & 0x80000000u;
  const uint64_t step = add2(pack2(__uint_as_float(s0 | 0x3F000000u), __uint_as_float(s1 | 0x3F000000u)), pack2(0.5f, 0.5f));   // 1 or 0
  return add2(step, pack2(__uint_as_float(__float_as_uint(u0) ^ s0), __uint_as_float(__float_as_uint(u1) ^ s1)));
}

// For calls that want sums that are not finite formed again: this warp's share of the accumulator, ahead of the epilogue that stores it
// and into the same places.  A pass of its own (a launch with such rows pays 0.1-1.2 us for it): the test inside the epilogues cost the
// fused activation of calls that have no use for it 2 %, and sending these calls through the row-by-row epilogue cost them 14 %.
__device__ __forceinline__ void redo_tile(const Params& P, uint32_t tmem_base, int acc, int q, int c0, int step, int lane, int64_t m0, int n0, int cols) {
  const int64_t row0 = m0 + q * 32;
  const bool row_ok = row0 + lane < P.M;
#pragma unroll 1
  for (int c = c0; c < cols / 32; c += step) {
    const int n = n0 + c * 32;
    if (n >= P.N) break;  // uniform
    const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + c * 32);
    uint32_t r[32];
    tmem_ld32(at, r);
    float zero = 0.f;
#pragma unroll
    for (int j = 0; j < 32; ++j) zero = fmaf(__uint_as_float(r[j]), 0.f, zero);
    if (!__any_sync(0xffffffffu, row_ok && zero != 0.f)) continue;
    float v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
    mst_redo_square<uint16_t>(P.redo, v, row0 + lane, row_ok, n, P.N);
#pragma unroll
    for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(v[j]);
    tmem_st32(at, r);
  }
}

// One 128 x BN accumulator (tensor-memory lanes = rows) -> rows of any leading dimension and alignment, for outputs the TMA
// unit cannot describe.  q = lane quarter this warp may read, m0/n0 = first row / column of this block's tile, c0 = first
// 32-column chunk this warp takes (the warps of one lane quarter interleave their chunks).  A chunk goes through the warp's
// staging box, so that a store instruction writes 32 neighbours of one row; stores by the row-owning lanes touch 32 lines
// each (2051 x 1999 bf16 outputs: 4.1 M two-byte stores to as many sectors).
// Activations (ACT) are taken behind the box too, so that the pre-activations travel as neighbours of one row.  By the row-owning lanes, two bytes to
// a line, 768 -> 3072 at 8192 tokens with pre-activations of odd pitch took 256 us for GELU and 99 for its derivative; now 49 and 69.  The
// derivative's are fetched a chunk ahead, a group of eight rows when the chunk before has used its own (eight rows ahead: 144 us).
template <int ACT, bool BF16>
__device__ __forceinline__ void epilogue_tile(const Params& P, uint32_t stage, uint32_t tmem_base, int acc, int q, int c0, int lane,
                                              int64_t m0, int n0, int split, int cols) {
  constexpr bool GRAD = ACT == MST_ACT_GELU_GRAD;
  constexpr int STEP = EPI_WARPS / 4;
  const int64_t row0 = (int64_t)m0 + q * 32;
  const uint32_t my_row = stage + (uint32_t)lane * 128u;
  const uint32_t sw = (uint32_t)(lane & 7);
  const int rows = P.M - row0 < 32 ? (int)(P.M - row0) : 32;
  uint16_t* const pre0 = reinterpret_cast<uint16_t*>(P.pre) + row0 * P.ldpre + lane;
  uint16_t x[GRAD ? 32 : 1];
  auto fetch = [&](int c, int r8) {
    const int n = n0 + c * 32;
    const bool any = c < cols / 32 && n + lane < P.N;
#pragma unroll
    for (int k = 0; k < 8; ++k) x[r8 + k] = any && r8 + k < rows ? pre0[n + (r8 + k) * P.ldpre] : (uint16_t)0;
  };
  if (GRAD) {
#pragma unroll
    for (int r8 = 0; r8 < 32; r8 += 8) fetch(c0, r8);
  }
#pragma unroll 1
  for (int c = c0; c < cols / 32; c += STEP) {
    const int n = n0 + c * 32;
    if (n >= P.N) break;  // uniform
    uint32_t r[32];
    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + c * 32), r);
    __syncwarp();  // the previous chunk has been read out of the box
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint32_t piece = (uint32_t)v ^ sw;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(my_row + piece * 16u), "r"(r[4 * v]), "r"(r[4 * v + 1]),
                   "r"(r[4 * v + 2]), "r"(r[4 * v + 3])
                   : "memory");
    }
    __syncwarp();
    const bool col_ok = n + lane < P.N;
    // A square inside the output is stored without a test per row (the branches and 64-bit addresses cost four times the stores).
    const bool inside = rows == 32 && n + 32 <= P.N;
    float* f32 = P.partial ? P.partial + (int64_t)split * P.M * P.N : reinterpret_cast<float*>(P.out);
    const int64_t ld = BF16 || !P.partial ? P.ldc : P.N;
    const int64_t at0 = row0 * ld + n + lane;
    auto group = [&](int r8) {
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) {   // eight rows are read back before the first is stored
        const uint32_t piece = (uint32_t)(lane >> 2) ^ (uint32_t)k;
        asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v[k]) : "r"(stage + (uint32_t)(r8 + k) * 128u + piece * 16u + (uint32_t)(lane & 3) * 4u) : "memory");
      }
      auto put = [&](uint16_t* to, int64_t pitch) {
        if (inside) {
#pragma unroll
          for (int k = 0; k < 8; ++k) to[k * pitch] = (uint16_t)(pack_bf16(v[k], 0.f) & 0xFFFFu);
        } else if (col_ok) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (r8 + k < rows) to[k * pitch] = (uint16_t)(pack_bf16(v[k], 0.f) & 0xFFFFu);
        }
      };
      if (GRAD) {
#pragma unroll
        for (int k = 0; k < 8; k += 2) {
          const uint64_t d = gelu_grad_pair(__uint_as_float((uint32_t)x[r8 + k] << 16), __uint_as_float((uint32_t)x[r8 + k + 1] << 16));
          unpack2(mul2(pack2(v[k], v[k + 1]), d), v[k], v[k + 1]);
        }
        fetch(c + STEP, r8);
      } else if (ACT == MST_ACT_GELU) {
        if (P.pre) put(pre0 + n + r8 * P.ldpre, P.ldpre);   // kept for the backward pass
#pragma unroll
        for (int k = 0; k < 8; k += 2) gelu_pair(v[k], v[k + 1]);
      }
      if (BF16) {
        put(reinterpret_cast<uint16_t*>(P.out) + at0 + r8 * ld, ld);
      } else {
        float* out = f32 + at0 + r8 * ld;
        if (inside) {
#pragma unroll
          for (int k = 0; k < 8; ++k) out[k * ld] = v[k];
        } else if (col_ok) {
#pragma unroll
          for (int k = 0; k < 8; ++k)
            if (r8 + k < rows) out[k * ld] = v[k];
        }
      }
    };
    if (GRAD) {
#pragma unroll
      for (int r8 = 0; r8 < 32; r8 += 8) group(r8);
    } else {
#pragma unroll 1
      for (int r8 = 0; r8 < rows; r8 += 8) group(r8);
    }
  }
}

// The sampled accumulator (weight gradient under the mask).  A chunk is 32 rows x one mask word; a warp's four chunks' words and
// CSR positions are fetched while the products still run (a wave's last tile has nothing else to hide them behind).  Chunks with
// few entries are written by the row-owning lanes, entry by entry.  Denser chunks turn from rows to columns through the warp's
// staging box, so that each store instruction writes the kept entries of ONE row, which are neighbours in CSR order; all 32 rows
// are read back before the first is stored, or every row would wait for its own round trip.
constexpr int SAMPLED_CHUNKS = BN / 32 / (EPI_WARPS / 4);
// Entries of a 1024-output chunk from which rows win: d of about 0.19.  8192 tokens, 768 x 768: entry by entry 15.5 / 16.6 / 19.3 /
// 24 us at d = 0.1 / 0.15 / 0.25 / 0.5, row by row 17.0 / 17.0 / 17.2 / 18.3.
constexpr int SAMPLED_STAGE_MIN = 192;
struct SampledWords {
  uint32_t word[SAMPLED_CHUNKS];
  int32_t at[SAMPLED_CHUNKS];
  __device__ __forceinline__ SampledWords(const Params& P, int q, int c0, int lane, int64_t m0, int n0) {
    const int64_t m = m0 + q * 32 + lane;
#pragma unroll
    for (int k = 0; k < SAMPLED_CHUNKS; ++k) {
      const int n = n0 + (c0 + k * (EPI_WARPS / 4)) * 32;
      word[k] = 0;
      at[k] = 0;
      if (m < P.M && n < P.N) {
        const int64_t wi = m * P.wpr + (n >> 5);
        word[k] = __ldg(P.bits + wi);
        at[k] = __ldg(P.wscan + wi);
      }
    }
  }
};
__device__ __forceinline__ void epilogue_tile_sampled(const Params& P, SampledWords W, uint32_t stage, uint32_t tmem_base, int acc,
                                                      int q, int c0, int lane, int n0, float* __restrict__ out) {
  const uint32_t my_row = stage + (uint32_t)lane * 128u;
  const uint32_t sw = (uint32_t)(lane & 7);
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll 1
  for (int k = 0; k < SAMPLED_CHUNKS; ++k) {   // rolled: four copies of this body cost the neighbouring launches instruction fetches
    const int c = c0 + k * (EPI_WARPS / 4);
    if (n0 + c * 32 >= P.N) break;  // uniform
    const uint32_t word = W.word[0];
    const int32_t at = W.at[0];
#pragma unroll
    for (int j = 1; j < SAMPLED_CHUNKS; ++j) {
      W.word[j - 1] = W.word[j];
      W.at[j - 1] = W.at[j];
    }
    uint32_t r[32];
    tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + c * 32), r);
    const int kept = __reduce_add_sync(0xFFFFFFFFu, __popc(word));
    if (kept < P.sampled_stage_min) {
      float* dst = out + at;
      int rank = 0;
#pragma unroll
      for (int j = 0; j < 32; ++j) {
        if ((word >> j) & 1u) {
          dst[rank] = __uint_as_float(r[j]);
          ++rank;
        }
      }
      continue;
    }
    __syncwarp();  // the previous chunk has been read out of the box
#pragma unroll
    for (int v = 0; v < 8; ++v) {
      const uint32_t piece = (uint32_t)v ^ sw;
      asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(my_row + piece * 16u), "r"(r[4 * v]), "r"(r[4 * v + 1]),
                   "r"(r[4 * v + 2]), "r"(r[4 * v + 3])
                   : "memory");
    }
    __syncwarp();
#pragma unroll
    for (int rr = 0; rr < 32; ++rr) {
      const uint32_t piece = (uint32_t)(lane >> 2) ^ (uint32_t)(rr & 7);
      asm volatile("ld.shared.b32 %0, [%1];" : "=r"(r[rr]) : "r"(stage + (uint32_t)rr * 128u + piece * 16u + (uint32_t)(lane & 3) * 4u) : "memory");
    }
#pragma unroll
    for (int rr = 0; rr < 32; ++rr) {
      const uint32_t w = __shfl_sync(0xFFFFFFFFu, word, rr);
      const int32_t base = __shfl_sync(0xFFFFFFFFu, at, rr);
      if ((w >> lane) & 1u) out[base + __popc(w & lt)] = __uint_as_float(r[rr]);
    }
  }
}

// eight fp32 values r[j..j+7] as bf16 into 16-byte piece `piece` of this lane's row of a staging box
__device__ __forceinline__ void stage_bf16(uint32_t my_row, uint32_t piece, const uint32_t (&r)[32], int j) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(my_row + piece * 16u),
               "r"(pack_bf16(__uint_as_float(r[j + 0]), __uint_as_float(r[j + 1]))),
               "r"(pack_bf16(__uint_as_float(r[j + 2]), __uint_as_float(r[j + 3]))),
               "r"(pack_bf16(__uint_as_float(r[j + 4]), __uint_as_float(r[j + 5]))),
               "r"(pack_bf16(__uint_as_float(r[j + 6]), __uint_as_float(r[j + 7])))
               : "memory");
}

// The TMA unit writes whole 16-byte pieces: of a row that ends inside one it would overwrite up to seven columns beyond, which are
// the caller's.  This lane's row of a box of 64 columns from n on: those behind the last whole piece.  Ahead of the fence that lets the box go.
__device__ __forceinline__ void store_tail(const Params& P, uint32_t my_row, uint32_t sw, void* out, int64_t ld, int64_t m, int n) {
  if (P.whole == P.N || P.whole >= n + 64 || m >= P.M) return;
  uint16_t* to = reinterpret_cast<uint16_t*>(out) + m * ld;
#pragma unroll 1
  for (int c = P.whole; c < P.N; ++c) {
    const uint32_t j = (uint32_t)(c - n);
    uint16_t v;
    asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(my_row + ((j >> 3) ^ sw) * 16u + (j & 7u) * 2u) : "memory");
    to[c] = v;
  }
}

// The same accumulator leaving through shared memory: each warp owns a 32-row x 128-byte staging box (128-byte
// swizzle: 16-byte piece j of row r sits at piece j ^ (r & 7), so the 32 row-owning lanes write without bank
// conflicts), fills it from its registers and one lane hands it to the TMA unit, which writes whole lines and clips
// rows >= M and columns >= N.  bf16: 64 columns per box (two tensor-memory reads); fp32: 32 columns per box, the
// K-range index as third coordinate.  Per-thread stores of a row-per-lane layout touch 32 lines per instruction and
// were measured to slow the concurrent main loop by about 15 %.
template <int KIND>
__device__ __forceinline__ void epilogue_tile_tma(const Params& P, const CUtensorMap* tmC, uint32_t stage, uint32_t tmem_base,
                                                  int acc, int q, int c0, int lane, int64_t m0, int n0, int split, int cols) {
  const int64_t row0 = (int64_t)m0 + q * 32;
  const uint32_t my_row = stage + (uint32_t)lane * 128u;
  const uint32_t sw = (uint32_t)(lane & 7);
  if (KIND != K_F32) {
#pragma unroll 1
    for (int g = c0; g < cols / 64; g += EPI_WARPS / 4) {
      const int n = n0 + g * 64;
      if (n >= P.N) break;  // uniform
      if (lane == 0) bulk_wait_read();  // the box's previous contents have left shared memory
      __syncwarp();
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        const int nn = n + h * 32;
        if (nn >= P.N) break;  // uniform; the TMA store clips these columns
        uint32_t r[32];
        tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + g * 64 + h * 32), r);
#pragma unroll
        for (int v = 0; v < 4; ++v) stage_bf16(my_row, (uint32_t)(h * 4 + v) ^ sw, r, 8 * v);
      }
      if (KIND == K_REDO) store_tail(P, my_row, sw, P.out, P.ldc, row0 + lane, n);
      fence_async_smem();
      __syncwarp();
      if (lane == 0 && row0 < P.M && (KIND != K_REDO || n < P.whole)) {
        tma_store_2d(tmC, stage, n, (int)row0);
        bulk_commit();
      }
    }
  } else {
#pragma unroll 1
    for (int c = c0; c < BN / 32; c += EPI_WARPS / 4) {
      const int n = n0 + c * 32;
      if (n >= P.N) break;  // uniform
      if (lane == 0) bulk_wait_read();
      __syncwarp();
      uint32_t r[32];
      tmem_ld32(tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + c * 32), r);
#pragma unroll
      for (int v = 0; v < 8; ++v) {
        const uint32_t piece = (uint32_t)v ^ sw;
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(my_row + piece * 16u), "r"(r[4 * v]), "r"(r[4 * v + 1]),
                     "r"(r[4 * v + 2]), "r"(r[4 * v + 3])
                     : "memory");
      }
      fence_async_smem();
      __syncwarp();
      if (lane == 0 && row0 < P.M) {
        tma_store_3d(tmC, stage, n, (int)row0, split);
        bulk_commit();
      }
    }
  }
}

// The bf16 accumulator with an activation.  Each warp has two boxes, so the pre-activation travels as whole lines too, and the two
// alternate: a box is filled while the other one's copy is on its way.  GELU: the accumulator goes to `box0` and, activated, to
// `box1`.  GELU_GRAD: the pre-activation of the warp's (at most two) 64-column groups is fetched into a box each, as soon as the
// tile before has left it, and each box turns into the result where it lies.
// The second box takes the place of one ring stage (0.8 us of 30).  GPT-2 small at 8192 tokens: fc1 with GELU and the pre-activation kept
// 47.0 -> 38.0 us (30.2 without the activation), fc2's input gradient with the derivative 53.5 -> 40.6 (30.2); a value at a time and the
// pre-activation row by row before.  Without the arithmetic the two take as long: what is left is the pre-activation's 50 MB.
struct ActBoxes {
  uint32_t box[2], bar[2];
  uint32_t phase;   // bit i: parity of the next filling of box i
};
__device__ __forceinline__ bool act_group(const Params& P, int c0, int i, int n0, int cols) {   // does the tile have the warp's group i?
  const int g = c0 + i * (EPI_WARPS / 4);
  return g < cols / 64 && n0 + g * 64 < P.N;
}
// one lane: the pre-activation of group i of a tile
__device__ __forceinline__ void fetch_pre(const Params& P, const CUtensorMap* tmP, const ActBoxes& A, int i, int q, int c0, int m0, int n0, int cols) {
  if (!act_group(P, c0, i, n0, cols)) return;
  mbar_expect_tx(A.bar[i], OUT_BOX_BYTES);
  tma_load_2d(A.box[i], tmP, n0 + (c0 + i * (EPI_WARPS / 4)) * 64, m0 + q * 32, A.bar[i]);
}
template <bool GRAD, bool TAIL>
__device__ __forceinline__ bool epilogue_tile_act(const Params& P, const CUtensorMap* tmC, const CUtensorMap* tmP, ActBoxes& A, uint32_t tmem_base, int acc,
                                                  int q, int c0, int lane, int64_t m0, int n0, int cols, volatile int* abort_flag) {
  const int64_t row0 = m0 + q * 32;
  const uint32_t sw = (uint32_t)(lane & 7);
#pragma unroll 1
  for (int i = 0; i < 2; ++i) {
    if (!act_group(P, c0, i, n0, cols)) break;  // uniform
    const int g = c0 + i * (EPI_WARPS / 4), n = n0 + g * 64;
    const uint32_t at = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(acc * BN + g * 64);
    if (GRAD) {
      const uint32_t my_row = (i ? A.box[1] : A.box[0]) + (uint32_t)lane * 128u;
      if (!mbar_wait(i ? A.bar[1] : A.bar[0], (A.phase >> i) & 1u, abort_flag)) return false;
      A.phase ^= 1u << i;
#pragma unroll 1
      for (int h = 0; h < 2; ++h) {
        uint32_t r[32], pw[16];
        tmem_ld32_nowait(at + (uint32_t)(h * 32), r);
#pragma unroll
        for (int v = 0; v < 4; ++v)
          asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(pw[4 * v]), "=r"(pw[4 * v + 1]), "=r"(pw[4 * v + 2]), "=r"(pw[4 * v + 3])
                       : "r"(my_row + (((uint32_t)(h * 4 + v)) ^ sw) * 16u));
        tmem_ld_wait(r);
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          const uint64_t d = gelu_grad_pair(__uint_as_float(pw[k] << 16), __uint_as_float(pw[k] & 0xFFFF0000u));
          float v0, v1;
          unpack2(mul2(pack2(r[2 * k], r[2 * k + 1]), d), v0, v1);
          r[2 * k] = __float_as_uint(v0);
          r[2 * k + 1] = __float_as_uint(v1);
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) stage_bf16(my_row, (uint32_t)(h * 4 + v) ^ sw, r, 8 * v);
      }
    } else {
      const uint32_t pre_row = A.box[0] + (uint32_t)lane * 128u, my_row = A.box[1] + (uint32_t)lane * 128u;
      uint32_t r[2][32];
      tmem_ld32_nowait(at, r[0]);
      tmem_ld32_nowait(at + 32u, r[1]);
      if (P.pre && lane == 0) bulk_wait_read_but_last();   // the pre-activations of the group before have left their box
      __syncwarp();
      tmem_ld_wait(r[0]);
      tmem_ld_wait(r[1]);
      if (P.pre) {                                         // kept for the backward pass
#pragma unroll
        for (int v = 0; v < 8; ++v) stage_bf16(pre_row, (uint32_t)v ^ sw, r[v >> 2], 8 * (v & 3));
        if (TAIL) store_tail(P, pre_row, sw, P.pre, P.ldpre, row0 + lane, n);
        fence_async_smem();
        __syncwarp();
        if (lane == 0) {
          if (row0 < P.M && (!TAIL || n < P.whole)) tma_store_2d(tmP, A.box[0], n, (int)row0);
          bulk_commit();
        }
      }
#pragma unroll
      for (int h = 0; h < 2; ++h) {
#pragma unroll
        for (int k = 0; k < 16; ++k) {
          float x0 = __uint_as_float(r[h][2 * k]), x1 = __uint_as_float(r[h][2 * k + 1]);
          gelu_pair(x0, x1);
          r[h][2 * k] = __float_as_uint(x0);
          r[h][2 * k + 1] = __float_as_uint(x1);
        }
        if (h == 0) {
          if (lane == 0) {
            if (P.pre) bulk_wait_read_but_last();          // the activations of the group before have
            else bulk_wait_read();
          }
          __syncwarp();
        }
#pragma unroll
        for (int v = 0; v < 4; ++v) stage_bf16(my_row, (uint32_t)(h * 4 + v) ^ sw, r[h], 8 * v);
      }
    }
    if (TAIL) store_tail(P, (GRAD && i == 0 ? A.box[0] : A.box[1]) + (uint32_t)lane * 128u, sw, P.out, P.ldc, row0 + lane, n);
    fence_async_smem();
    __syncwarp();
    if (lane == 0) {
      if (row0 < P.M && (!TAIL || n < P.whole)) tma_store_2d(tmC, GRAD && i == 0 ? A.box[0] : A.box[1], n, (int)row0);
      bulk_commit();
    }
  }
  return true;
}
// GELU_GRAD, one lane: the next tile's pre-activations, each into its box when this tile's copy has read it
__device__ __forceinline__ void fetch_next(const Params& P, const CUtensorMap* tmP, const ActBoxes& A, int q, int c0, int n0, int cols, int next_m0, int next_n0,
                                           int next_cols) {
  if (act_group(P, c0, 1, n0, cols)) bulk_wait_read_but_last();
  else bulk_wait_read();
  fetch_pre(P, tmP, A, 0, q, c0, next_m0, next_n0, next_cols);
  bulk_wait_read();
  fetch_pre(P, tmP, A, 1, q, c0, next_m0, next_n0, next_cols);
}

// ------------------------------------------------------------------------------------------- kernel
template <int KIND>
__global__ void __launch_bounds__(NUM_THREADS, 1)
tc_gemm_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
               const __grid_constant__ CUtensorMap tmC, const __grid_constant__ CUtensorMap tmP, const Params P) {
  const bool A_MN = P.major == M_GRADIENT, B_MN = P.major != M_FORWARD;
  constexpr bool ACT = KIND == K_ACT || KIND == K_REDO_ACT, REDO = KIND == K_REDO || KIND == K_REDO_ACT;
  constexpr int RING = STAGES - (ACT ? 1 : 0);
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles_base = (raw + 1023u) & ~1023u;  // swizzled tiles need 1024-byte alignment
  const uint32_t out_base = tiles_base + STAGES * STAGE_BYTES;  // epilogue staging boxes (1024-byte aligned)
  const uint32_t bar_base = out_base + EPI_WARPS * OUT_BOX_BYTES;
  // barrier slots (8 bytes each): full[STAGES], empty[STAGES], tmem_full[2], tmem_empty[2], pre_full[2 * EPI_WARPS]
  const uint32_t full0 = bar_base, empty0 = bar_base + 8 * STAGES, tfull0 = bar_base + 16 * STAGES,
                 tempty0 = tfull0 + 16, pre0 = tempty0 + 16;
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, EPI_WARPS);
    }
    for (int e = 0; e < 2 * EPI_WARPS; ++e) mbar_init(pre0 + 8 * e, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();  // set-up above overlaps the predecessor's tail; global memory only from here on

  const int64_t works = (int64_t)P.m_tiles * P.n_tiles * P.splits;
  const int tiles = P.m_tiles * P.n_tiles;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      for (int64_t w = blockIdx.x; w < works && !*abort_flag; w += gridDim.x) {
        const int split = (int)(w / tiles), t = (int)(w % tiles);
        const int m0 = (t / P.n_tiles) * BM, n0 = (t % P.n_tiles) * BN;
        const int kb0 = (int)((int64_t)split * P.kblocks / P.splits), kb1 = (int)((int64_t)(split + 1) * P.kblocks / P.splits);
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag)) break;
          const uint32_t fb = full0 + 8 * s;
          const uint32_t sa = tiles_base + s * STAGE_BYTES, sb = sa + A_BYTES;
          mbar_expect_tx(fb, STAGE_BYTES);
          if (A_MN) {
            for (int j = 0; j < BM / 64; ++j) tma_load_2d(sa + j * BOX_BYTES, &tmA, m0 + j * 64, kb * BK, fb);
          } else {
            tma_load_2d(sa, &tmA, kb * BK, m0, fb);
          }
          if (B_MN) {
            for (int j = 0; j < BN / 64; ++j) tma_load_2d(sb + j * BOX_BYTES, &tmB, n0 + j * 64, kb * BK, fb);
          } else {
            tma_load_2d(sb, &tmB, kb * BK, n0, fb);
          }
          if (++s == RING) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      // instruction descriptor: fp32 accumulate, bf16 x bf16, M = 128, N = 256, operand majors
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(A_MN ? 1 : 0) << 15) |
                             ((uint32_t)(B_MN ? 1 : 0) << 16) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(BM >> 4) << 24);
      // The issue loop is one thread's serial instruction stream; everything that does not depend on the stage is
      // formed once here.  K-major: 16 K-elements = 32 bytes further along the swizzled row; MN-major: 16 rows of
      // 128 bytes.
      const uint64_t adesc0 = smem_desc(tiles_base, A_MN ? BOX_BYTES : 16, 1024);
      const uint64_t bdesc0 = smem_desc(tiles_base + A_BYTES, B_MN ? BOX_BYTES : 16, 1024);
      const uint32_t a_kstep = (uint32_t)(A_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      const uint32_t b_kstep = (uint32_t)(B_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      int s = 0, acc = 0;
      uint32_t ph = 0, acc_ph = 0;
      for (int64_t w = blockIdx.x; w < works && !*abort_flag; w += gridDim.x) {
        const int split = (int)(w / tiles);
        const int kb0 = (int)((int64_t)split * P.kblocks / P.splits), kb1 = (int)((int64_t)(split + 1) * P.kblocks / P.splits);
        if (!mbar_wait(tempty0 + 8 * acc, acc_ph ^ 1u, abort_flag)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          // descriptors of this stage: the start-address field moves by 16-byte units, nothing else changes
          const uint64_t ad = adesc0 + (uint64_t)(uint32_t)(s * (STAGE_BYTES >> 4));
          const uint64_t bd = bdesc0 + (uint64_t)(uint32_t)(s * (STAGE_BYTES >> 4));
          tc_mma(d_tmem, ad, bd, idesc, kb > kb0 ? 1u : 0u);
#pragma unroll
          for (int k = 1; k < BK / UMMA_K; ++k) tc_mma(d_tmem, ad + (uint64_t)(k * a_kstep), bd + (uint64_t)(k * b_kstep), idesc, 1u);
          tc_commit(empty0 + 8 * s);  // the smem stage is free once these MMAs have read it
          if (++s == RING) { s = 0; ph ^= 1u; }
        }
        if (!ok) break;
        tc_commit(tfull0 + 8 * acc);  // accumulator complete
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (warps 2..9)
    const int q = warp & 3;  // tensor-memory lane quarter this warp may read
    const bool fetch = ACT && P.act == MST_ACT_GELU_GRAD;
    const int c0 = (warp - 2) >> 2;   // the warps of a lane quarter interleave their chunks
    const uint32_t box = out_base + (uint32_t)(warp - 2) * OUT_BOX_BYTES, box1 = tiles_base + (uint32_t)((STAGES - 1) * STAGE_BYTES + (warp - 2) * OUT_BOX_BYTES);
    ActBoxes A = {{box, box1}, {pre0 + 16 * (warp - 2), pre0 + 16 * (warp - 2) + 8}, 0};
    int acc = 0;
    uint32_t acc_ph = 0;
    for (int64_t w = blockIdx.x; w < works; w += gridDim.x) {
      const int split = (int)(w / tiles), t = (int)(w % tiles);
      const int m0 = (t / P.n_tiles) * BM, n0 = (t % P.n_tiles) * BN;
      if (KIND == K_SAMPLED) {
        const SampledWords W(P, q, c0, lane, m0, n0);
        if (!mbar_wait(tfull0 + 8 * acc, acc_ph, abort_flag)) break;
        tc_fence_after();
        epilogue_tile_sampled(P, W, box, tmem_base, acc, q, c0, lane, n0,
                              P.partial ? P.partial + (int64_t)split * P.nnz : reinterpret_cast<float*>(P.out));
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(tempty0 + 8 * acc);
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
        continue;
      }
      if (fetch && lane == 0 && w == blockIdx.x) {
        fetch_pre(P, &tmP, A, 0, q, c0, m0, n0, BN);
        fetch_pre(P, &tmP, A, 1, q, c0, m0, n0, BN);
      }
      if (!mbar_wait(tfull0 + 8 * acc, acc_ph, abort_flag)) break;
      tc_fence_after();
      if (REDO && P.redo.kind) {   // the chunks this warp stores: pairs of them
        redo_tile(P, tmem_base, acc, q, 2 * c0, EPI_WARPS / 2, lane, m0, n0, BN);
        redo_tile(P, tmem_base, acc, q, 2 * c0 + 1, EPI_WARPS / 2, lane, m0, n0, BN);
      }
      if (ACT) {
        if (!(P.major == M_INPUT ? epilogue_tile_act<true, REDO>(P, &tmC, &tmP, A, tmem_base, acc, q, c0, lane, m0, n0, BN, abort_flag)
                                 : epilogue_tile_act<false, REDO>(P, &tmC, &tmP, A, tmem_base, acc, q, c0, lane, m0, n0, BN, abort_flag)))
          break;
        if (fetch && lane == 0 && w + gridDim.x < works) {
          const int tn = (int)((w + gridDim.x) % tiles);
          fetch_next(P, &tmP, A, q, c0, n0, BN, (tn / P.n_tiles) * BM, (tn % P.n_tiles) * BN, BN);
        }
      } else if (KIND != K_ROWS && KIND != K_ROWS_ACT) {
        epilogue_tile_tma<KIND>(P, &tmC, box, tmem_base, acc, q, c0, lane, m0, n0, split, BN);
      } else {
        if (P.redo.kind) redo_tile(P, tmem_base, acc, q, c0, EPI_WARPS / 4, lane, m0, n0, BN);
        if (KIND == K_ROWS && P.major == M_GRADIENT) epilogue_tile<MST_ACT_NONE, false>(P, box, tmem_base, acc, q, c0, lane, m0, n0, split, BN);
        else if (KIND == K_ROWS) epilogue_tile<MST_ACT_NONE, true>(P, box, tmem_base, acc, q, c0, lane, m0, n0, split, BN);
        else if (P.major == M_INPUT) epilogue_tile<MST_ACT_GELU_GRAD, true>(P, box, tmem_base, acc, q, c0, lane, m0, n0, split, BN);
        else epilogue_tile<MST_ACT_GELU, true>(P, box, tmem_base, acc, q, c0, lane, m0, n0, split, BN);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty0 + 8 * acc);
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
    if (KIND != K_SAMPLED && KIND != K_ROWS && KIND != K_ROWS_ACT && lane == 0) bulk_wait_read();  // this warp's stores have left shared memory; the end of the grid waits for their arrival
  }

  // ------------------------------------------------------------------ teardown
  if (*abort_flag) {
    // give copies and MMAs already in flight time to land before shared and tensor memory are released
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// ------------------------------------------------------------------------------------------- CTA-pair kernel
// Same roles, but two blocks of a cluster (an SM pair) share one 256 x 256 output tile: each block loads its own 128
// rows of A and its own half (128 of 256 columns) of B, the even block issues tcgen05.mma.cta_group::2 (M = 256) that
// reads both blocks' shared memory and writes both blocks' tensor memory.  Per block this halves the shared-memory
// traffic for B, which is what bounds the single-block kernel.  Barrier protocol:
//   full[s]   (even block)  two arrivals (one per block's producer, each announcing its own bytes) + TMA bytes of both
//   empty[s]  (each block)  one arrival, multicast by the even block's tcgen05.commit
//   tfull[a]  (each block)  one arrival, multicast by tcgen05.commit after the tile's last MMA
//   tempty[a] (even block)  sixteen arrivals: the eight epilogue warps of both blocks
constexpr int P_STAGES = 6;
constexpr int PB_BYTES = (BN / 2) * BK * 2;        // this block's half of B: 16 KiB
constexpr int P_STAGE_BYTES = A_BYTES + PB_BYTES;  // 32 KiB
constexpr size_t P_SMEM_BYTES = (size_t)P_STAGES * P_STAGE_BYTES + EPI_WARPS * OUT_BOX_BYTES + 1024 + 256;
// The jobs of a pair, one after the other: a tile's rows and columns over one K range.  Jobs beyond P.full, a last wave that would
// leave at least half of the pairs idle, are cut into P.cut:
//   products with the weights (rows of bf16)   two halves of the tile's columns; a tile whose columns end within its first half is
//                                              half as wide in any case;
//   gradients                                  parts of the job's K range, with sums (`split`) of their own.
// (The k-blocks of all tiles shared out evenly were slower, 34 -> 40 us for 2304 x 768 at 8192 tokens and 108 -> 144 for 4096 x 1024
// at 16384: pairs at different places of the K range read the activations at different times, and L2 does not hold them.)
template <int KIND>
struct PairJobs {
  uint32_t w, end, step, tiles;
  int split, m0, n0, cols, kb0, kb1;
  __device__ __forceinline__ PairJobs(const Params& P, uint32_t pair, uint32_t npairs) {
    tiles = (uint32_t)((P.m_tiles + 1) / 2) * (uint32_t)P.n_tiles;
    w = pair;
    end = P.full + P.cut * (tiles * (uint32_t)P.splits - P.full);
    step = npairs;
    split = kb0 = 0;
    kb1 = P.kblocks;
  }
  __device__ __forceinline__ bool next(const Params& P) {
    while (w < end) {
      uint32_t job = w, part = 0;
      const bool cut = w >= P.full;
      if (cut) {
        const uint32_t k = w - P.full;
        job = P.full + k / P.cut;
        part = k - (job - P.full) * P.cut;
      }
      w += step;
      uint32_t tile = job, range = 0;
      if (job >= tiles) {
        range = job / tiles;
        tile = job - range * tiles;
      }
      const uint32_t row = tile / (uint32_t)P.n_tiles;
      m0 = (int)row * (2 * BM);
      n0 = (int)(tile - row * (uint32_t)P.n_tiles) * BN;
      if (KIND == K_BF16 || KIND == K_ACT || KIND == K_REDO || KIND == K_REDO_ACT || KIND == K_ROWS_ACT || (KIND == K_ROWS && P.epilogue == MST_TC_OUT_BF16)) {
        n0 += (int)part * (BN / 2);
        cols = cut || P.N - n0 <= BN / 2 ? BN / 2 : BN;
        if (n0 >= P.N) continue;   // that half lies outside the output
      } else {
        cols = BN;
        if (P.splits > 1 || cut) {
          kb0 = (int)((int64_t)range * P.kblocks / P.splits);
          kb1 = (int)((int64_t)(range + 1) * P.kblocks / P.splits);
          split = (int)(range + part);
          if (cut) {
            const int n = kb1 - kb0, from = kb0;
            kb0 = from + (int)((int64_t)part * n / P.cut);
            kb1 = from + (int)((int64_t)(part + 1) * n / P.cut);
          }
        }
      }
      return true;
    }
    return false;
  }
};
// shared::cluster address of the same shared-memory location in the even block (rank 0) of the pair
__device__ __forceinline__ uint32_t in_even_block(uint32_t local_addr) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(local_addr), "r"(0u));
  return r;
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx_cluster(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cluster.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* tm, int x, int y, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
      "l"(tm), "r"(x), "r"(y), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void tc_mma_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accum) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accum)
      : "memory");
}
__device__ __forceinline__ void tc_commit_pair(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
               "h"((uint16_t)3)
               : "memory");
}

template <int KIND, int MAJOR>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(NUM_THREADS, 1)
tc_gemm_pair_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const __grid_constant__ CUtensorMap tmBn, const __grid_constant__ CUtensorMap tmC,
                    const __grid_constant__ CUtensorMap tmP, const Params P) {
  constexpr bool A_MN = MAJOR == M_GRADIENT, B_MN = MAJOR != M_FORWARD;
  constexpr bool ACT = KIND == K_ACT || KIND == K_REDO_ACT, REDO = KIND == K_REDO || KIND == K_REDO_ACT;
  constexpr int RING = P_STAGES - (ACT ? 1 : 0);
  extern __shared__ unsigned char smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t tiles_base = (raw + 1023u) & ~1023u;
  const uint32_t out_base = tiles_base + P_STAGES * P_STAGE_BYTES;
  const uint32_t bar_base = out_base + EPI_WARPS * OUT_BOX_BYTES;
  const uint32_t full0 = bar_base, empty0 = bar_base + 8 * P_STAGES, tfull0 = bar_base + 16 * P_STAGES,
                 tempty0 = tfull0 + 16, pre0 = tempty0 + 16;
  __shared__ uint32_t tmem_base_holder;
  __shared__ int abort_sh;
  volatile int* abort_flag = &abort_sh;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();  // 0 = even block (issues the MMAs), 1 = its peer
  if (threadIdx.x == 0) {
    abort_sh = 0;
    for (int s = 0; s < P_STAGES; ++s) {
      mbar_init(full0 + 8 * s, 2);
      mbar_init(empty0 + 8 * s, 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(tfull0 + 8 * a, 1);
      mbar_init(tempty0 + 8 * a, 2 * EPI_WARPS);
    }
    for (int e = 0; e < 2 * EPI_WARPS; ++e) mbar_init(pre0 + 8 * e, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0 && lane < 4)   // the maps are parameters: fetched while the predecessor drains
    asm volatile("prefetch.tensormap [%0];" ::"l"(lane == 0 ? &tmA : lane == 1 ? &tmB : lane == 2 ? &tmBn : &tmC) : "memory");
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_base_holder)),
                 "r"(TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // both blocks' barriers are initialised before any remote arrival or copy completion
  tc_fence_after();
  const uint32_t tmem_base = tmem_base_holder;
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();

  const uint32_t pair = blockIdx.x >> 1, npairs = gridDim.x >> 1;

  if (warp == 0) {
    // ------------------------------------------------------------------ producer (both blocks)
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0;
      PairJobs<KIND> J(P, pair, npairs);
      while (J.next(P) && !*abort_flag) {
        const int m0 = J.m0 + (int)rank * BM;              // this block's rows
        const int n0 = J.n0 + (int)rank * (J.cols / 2);    // this block's half of B
        const uint32_t bytes = (uint32_t)(A_BYTES + J.cols / 2 * BK * 2);
        const int kb0 = J.kb0, kb1 = J.kb1;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(empty0 + 8 * s, ph ^ 1u, abort_flag)) break;
          const uint32_t fb = in_even_block(full0 + 8 * s);  // the even block's barrier collects both blocks' bytes
          const uint32_t sa = tiles_base + s * P_STAGE_BYTES, sb = sa + A_BYTES;
          mbar_expect_tx_cluster(fb, bytes);
          if (A_MN) {
            for (int j = 0; j < BM / 64; ++j) tma_load_2d_pair(sa + j * BOX_BYTES, &tmA, m0 + j * 64, kb * BK, fb);
          } else {
            tma_load_2d_pair(sa, &tmA, kb * BK, m0, fb);
          }
          if (B_MN) {
            tma_load_2d_pair(sb, &tmB, n0, kb * BK, fb);
            if (J.cols == BN) tma_load_2d_pair(sb + BOX_BYTES, &tmB, n0 + 64, kb * BK, fb);
          } else {
            tma_load_2d_pair(sb, J.cols == BN ? &tmB : &tmBn, kb * BK, n0, fb);
          }
          if (++s == RING) { s = 0; ph ^= 1u; }
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------ MMA issuer (even block only)
    if (lane == 0 && rank == 0) {
      const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(A_MN ? 1 : 0) << 15) |
                              ((uint32_t)(B_MN ? 1 : 0) << 16) | ((uint32_t)((2 * BM) >> 4) << 24);
      const uint64_t adesc0 = smem_desc(tiles_base, A_MN ? BOX_BYTES : 16, 1024);
      const uint64_t bdesc0 = smem_desc(tiles_base + A_BYTES, B_MN ? BOX_BYTES : 16, 1024);
      const uint32_t a_kstep = (uint32_t)(A_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      const uint32_t b_kstep = (uint32_t)(B_MN ? UMMA_K * 128 : UMMA_K * 2) >> 4;
      int s = 0, acc = 0;
      uint32_t ph = 0, acc_ph = 0;
      PairJobs<KIND> J(P, pair, npairs);
      while (J.next(P) && !*abort_flag) {
        const uint32_t idesc = idesc0 | ((uint32_t)(J.cols >> 3) << 17);
        const int kb0 = J.kb0, kb1 = J.kb1;
        if (!mbar_wait(tempty0 + 8 * acc, acc_ph ^ 1u, abort_flag)) break;
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + (uint32_t)(acc * BN);
        bool ok = true;
        for (int kb = kb0; kb < kb1; ++kb) {
          if (!mbar_wait(full0 + 8 * s, ph, abort_flag)) { ok = false; break; }
          tc_fence_after();
          // descriptors of this stage: the start-address field moves by 16-byte units, nothing else changes
          const uint64_t ad = adesc0 + (uint64_t)(uint32_t)(s * (P_STAGE_BYTES >> 4));
          const uint64_t bd = bdesc0 + (uint64_t)(uint32_t)(s * (P_STAGE_BYTES >> 4));
          tc_mma_pair(d_tmem, ad, bd, idesc, kb > kb0 ? 1u : 0u);
#pragma unroll
          for (int k = 1; k < BK / UMMA_K; ++k) tc_mma_pair(d_tmem, ad + (uint64_t)(k * a_kstep), bd + (uint64_t)(k * b_kstep), idesc, 1u);
          tc_commit_pair(empty0 + 8 * s);  // frees this stage in both blocks
          if (++s == RING) { s = 0; ph ^= 1u; }
        }
        if (!ok) break;
        tc_commit_pair(tfull0 + 8 * acc);  // both blocks' halves of the accumulator are complete
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
      }
    }
  } else {
    // ------------------------------------------------------------------ epilogue (both blocks, own 128 rows)
    const int q = warp & 3;
    const bool fetch = ACT && P.act == MST_ACT_GELU_GRAD;
    const int c0 = (warp - 2) >> 2;   // the warps of a lane quarter interleave their chunks
    const uint32_t box = out_base + (uint32_t)(warp - 2) * OUT_BOX_BYTES, box1 = tiles_base + (uint32_t)((P_STAGES - 1) * P_STAGE_BYTES + (warp - 2) * OUT_BOX_BYTES);
    ActBoxes A = {{box, box1}, {pre0 + 16 * (warp - 2), pre0 + 16 * (warp - 2) + 8}, 0};
    int acc = 0;
    uint32_t acc_ph = 0;
    PairJobs<KIND> J(P, pair, npairs);
    bool first = true;
    while (J.next(P)) {
      const int m0 = J.m0 + (int)rank * BM, n0 = J.n0;
      const int split = J.split;
      if (KIND == K_SAMPLED) {
        const SampledWords W(P, q, c0, lane, m0, n0);
        if (!mbar_wait(tfull0 + 8 * acc, acc_ph, abort_flag)) break;
        tc_fence_after();
        epilogue_tile_sampled(P, W, box, tmem_base, acc, q, c0, lane, n0,
                              P.partial ? P.partial + (int64_t)split * P.nnz : reinterpret_cast<float*>(P.out));
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(in_even_block(tempty0 + 8 * acc));
        if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
        continue;
      }
      if (fetch && lane == 0 && first) {
        fetch_pre(P, &tmP, A, 0, q, c0, m0, n0, J.cols);
        fetch_pre(P, &tmP, A, 1, q, c0, m0, n0, J.cols);
      }
      first = false;
      if (!mbar_wait(tfull0 + 8 * acc, acc_ph, abort_flag)) break;
      tc_fence_after();
      if (REDO && P.redo.kind) {   // the chunks this warp stores: pairs of them
        redo_tile(P, tmem_base, acc, q, 2 * c0, EPI_WARPS / 2, lane, m0, n0, J.cols);
        redo_tile(P, tmem_base, acc, q, 2 * c0 + 1, EPI_WARPS / 2, lane, m0, n0, J.cols);
      }
      if (ACT) {
        if (!epilogue_tile_act<MAJOR == M_INPUT, REDO>(P, &tmC, &tmP, A, tmem_base, acc, q, c0, lane, m0, n0, J.cols, abort_flag)) break;
        if (fetch) {
          PairJobs<KIND> N = J;
          if (N.next(P) && lane == 0) fetch_next(P, &tmP, A, q, c0, n0, J.cols, N.m0 + (int)rank * BM, N.n0, N.cols);
        }
      } else if (KIND != K_ROWS && KIND != K_ROWS_ACT) {
        epilogue_tile_tma<KIND>(P, &tmC, box, tmem_base, acc, q, c0, lane, m0, n0, split, J.cols);
      } else {
        if (P.redo.kind) redo_tile(P, tmem_base, acc, q, c0, EPI_WARPS / 4, lane, m0, n0, J.cols);
        epilogue_tile<KIND == K_ROWS ? MST_ACT_NONE : MAJOR == M_INPUT ? MST_ACT_GELU_GRAD : MST_ACT_GELU, MAJOR != M_GRADIENT>(P, box, tmem_base, acc, q, c0, lane, m0, n0, split, J.cols);
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(in_even_block(tempty0 + 8 * acc));
      if (++acc == 2) { acc = 0; acc_ph ^= 1u; }
    }
    if (KIND != K_SAMPLED && KIND != K_ROWS && KIND != K_ROWS_ACT && lane == 0) bulk_wait_read();  // this warp's stores have left shared memory; the end of the grid waits for their arrival
  }

  // ------------------------------------------------------------------ teardown
  if (*abort_flag) {
    for (int i = 0; i < 2000; ++i) __nanosleep(1000);
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();  // the peer may still be signalling this block's barriers or reading its shared memory
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(TMEM_COLS) : "memory");
  }
}

// out[i] = sum over splits of partial[s][i], fixed order
__global__ void tc_reduce_kernel(const float* __restrict__ partial, int splits, int64_t n, float* __restrict__ out) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float s = partial[i];
  for (int k = 1; k < splits; ++k) s += partial[(int64_t)k * n + i];
  out[i] = s;
}

// the same, four values per thread (n a multiple of 4, 16-byte aligned pointers)
__global__ void tc_reduce4_kernel(const float4* __restrict__ partial, int splits, int64_t n4, float4* __restrict__ out) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n4) return;
  float4 s = partial[i];
  for (int k = 1; k < splits; ++k) {
    const float4 v = partial[(int64_t)k * n4 + i];
    s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
  }
  out[i] = s;
}

// The same where the last jobs were cut, so that tiles have different numbers of sums: a warp per row of a tile.  Sampled output: the
// row's kept entries are one run.
__global__ void __launch_bounds__(256) tc_reduce_tiles_kernel(const Params P) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int lane = threadIdx.x & 31;
  const int64_t m = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int g = blockIdx.y;
  if (m >= P.M) return;
  const uint32_t tiles = (uint32_t)((P.m_tiles + 1) / 2) * (uint32_t)P.n_tiles, t = (uint32_t)(m / (2 * BM)) * (uint32_t)P.n_tiles + (uint32_t)g;
  const int sums = P.splits + (t + (uint32_t)(P.splits - 1) * tiles >= P.full ? (int)P.cut - 1 : 0);
  int64_t first, last, slab;
  const float* in = P.partial;
  float* out = reinterpret_cast<float*>(P.out);
  if (P.epilogue == MST_TC_OUT_SAMPLED) {
    const int64_t w0 = m * P.wpr + g * (BN / 32);
    first = P.wscan[w0];
    last = P.wscan[(g + 1) * (BN / 32) < P.wpr ? w0 + BN / 32 : (m + 1) * P.wpr];
    slab = P.nnz;
  } else {
    first = (int64_t)g * BN;
    last = first + BN < P.N ? first + BN : P.N;
    slab = P.M * P.N;
    in += m * P.N;
    out += m * P.ldc;
  }
  for (int64_t e = first + lane; e < last; e += 32) {
    float v = in[e];
    for (int k = 1; k < sums; ++k) v += in[k * slab + e];
    out[e] = v;
  }
}

// The same for a dense gradient whose entries under the mask are wanted as well (regrowth steps): four columns per lane, a warp per
// 128 columns of a row; the sums go to both places (4 us less per layer of a GPT-2-small block than a pass over the result).
__global__ void __launch_bounds__(256) tc_reduce_sample_kernel(const Params P, float* __restrict__ dW) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int lane = threadIdx.x & 31;
  const int64_t m = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), c = (int64_t)blockIdx.y * 128 + lane * 4;
  if (m >= P.M || c >= P.N) return;
  const uint32_t tiles = (uint32_t)((P.m_tiles + 1) / 2) * (uint32_t)P.n_tiles, t = (uint32_t)(m / (2 * BM)) * (uint32_t)P.n_tiles + (uint32_t)(c / BN);
  const int sums = P.splits + (t + (uint32_t)(P.splits - 1) * tiles >= P.full ? (int)P.cut - 1 : 0);
  const int64_t wi = m * P.wpr + (c >> 5);
  const uint32_t word = __ldg(P.bits + wi), sh = (uint32_t)c & 31u;
  const int32_t first = __ldg(P.wscan + wi);
  const float* in = P.partial + m * P.N + c;
  float4 v = *reinterpret_cast<const float4*>(in);
  for (int k = 1; k < sums; ++k) {
    const float4 x = *reinterpret_cast<const float4*>(in + k * P.M * P.N);
    v.x += x.x; v.y += x.y; v.z += x.z; v.w += x.w;
  }
  *reinterpret_cast<float4*>(reinterpret_cast<float*>(P.out) + m * P.ldc + c) = v;
  const uint32_t nib = (word >> sh) & 15u;
  float* d = dW + first + __popc(word & ((1u << sh) - 1u));
  if (nib & 1u) d[0] = v.x;
  if (nib & 2u) d[__popc(nib & 1u)] = v.y;
  if (nib & 4u) d[__popc(nib & 3u)] = v.z;
  if (nib & 8u) d[__popc(nib & 7u)] = v.w;
}

// ------------------------------------------------------------------------------------------- host side
// rows x cols (cols contiguous, ld elements between rows) bf16 matrix; box = box_rows x 64 columns
bool make_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t cols, int64_t ld, int box_rows) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64u, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Output maps for the staged epilogue.  bf16 [M x N] (ld elements between rows), box 64 columns x 32 rows;
// fp32 [splits x M x N], box 32 columns x 32 rows x 1.  Both boxes are 128 bytes wide (128-byte swizzle).
bool make_out_map_bf16(CUtensorMap* tm, void* base, int64_t M, int64_t N, int64_t ld) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn || (ld % 8) != 0 || (reinterpret_cast<uintptr_t>(base) & 15u) != 0) return false;
  cuuint64_t dims[2] = {(cuuint64_t)N, (cuuint64_t)M};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {64u, 32u};
  cuuint32_t estr[2] = {1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
bool make_out_map_f32(CUtensorMap* tm, void* base, int64_t M, int64_t N, int64_t ld, int64_t slab_elems, int splits) {
  mst_encode_tiled_fn fn = mst_encode_tiled();
  if (!fn || (ld % 4) != 0 || (slab_elems % 4) != 0 || (reinterpret_cast<uintptr_t>(base) & 15u) != 0) return false;
  cuuint64_t dims[3] = {(cuuint64_t)N, (cuuint64_t)M, (cuuint64_t)splits};
  cuuint64_t strides[2] = {(cuuint64_t)ld * 4, (cuuint64_t)slab_elems * 4};
  cuuint32_t box[3] = {32u, 32u, 1u};
  cuuint32_t estr[3] = {1u, 1u, 1u};
  return fn(tm, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, base, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_NONE, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

mst_encode_tiled_fn mst_encode_tiled() {
  static mst_encode_tiled_fn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (mst_encode_tiled_fn)p;
  }
  return fn;
}

int mst_sm_count() {
  static int n[64] = {};
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev < 0 || dev >= 64) return 148;
  if (!n[dev]) {
    if (cudaDeviceGetAttribute(&n[dev], cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n[dev] <= 0) n[dev] = 148;
  }
  return n[dev];
}

// Number of K ranges for a contraction whose output has few tiles, and into how many parts (*cut, 1: none) the jobs of a last wave
// that would leave half of the slots idle are cut when there is one range (cutting the last of several ranges lost: 2304 x 768
// at 8192 tokens 34 -> 41 us, 1280 x 1280 at 16384 70 -> 84): minimise a simple time model
//   waves * (k-blocks per range * t_kblock + t_tile) + traffic of the partial sums
// over 1..16 ranges.  `tiles` of the output, `slots` = jobs that run at once (blocks or block pairs), `out_bytes` = bytes one range
// writes as partial sums (and the reduction reads back).  75 tiles on 74 pairs (3840 x 1280, 16384
// tokens, d = 0.5) are one wave and a sixteenth, 171 us; without the cut they were three waves of two ranges, 185 us.
int mst_tc_pick_splits(int64_t tiles, int64_t slots, int64_t kblocks, double out_bytes, int* cut) {
  const double t_kblock = 0.32e-6, t_tile = 1.5e-6, bw = 4.0e12, t_reduce_launch = 3.0e-6;
  int best = 1;
  double best_t = 1e30;
  *cut = 1;
  for (int sp = 1; sp <= 16 && sp <= kblocks; ++sp) {
    const int64_t jobs = tiles * sp, rest = jobs % slots, waves = (jobs + slots - 1) / slots;
    const double kb = (double)((kblocks + sp - 1) / sp);
    double t = (double)waves * (kb * t_kblock + t_tile);
    if (sp > 1) t += t_reduce_launch + (double)sp * out_bytes * 2.0 / bw;
    int c = 1;
    if (sp == 1 && rest > 0 && jobs > slots && rest * 2 <= slots) {
      int parts = (int)(slots / rest < 16 ? slots / rest : 16);
      while (parts > 1 && kb / parts < 4.0) --parts;
      const double sums = 1.0 + (double)rest * (parts - 1) / (double)tiles;
      const double tc = (double)(waves - 1) * (kb * t_kblock + t_tile) + kb / parts * t_kblock + 3.0 * t_tile + t_reduce_launch + sums * out_bytes * 2.0 / bw;
      if (parts > 1 && tc < t * 0.95) { t = tc; c = parts; }
    }
    if (t < best_t * 0.97) {  // prefer fewer ranges unless the gain is clear
      best_t = t;
      best = sp;
      *cut = c;
    }
  }
  return best;
}

// Per-device scratch buffers, grown on demand (growing waits for the device and frees the old buffer).
//   MST_WS_SPLIT    partial sums of a K-range split.  Every call that splits its contraction range shares its device's
//                   buffer, so two such calls must not overlap on the GPU (mst_dense_grad, mst_dense_grad_dw,
//                   mst_sddmm_dw and the host-step calls on the tensor path): keep them on one stream or order them
//                   with events.
//   MST_WS_COLUMNS  operands prepared for one call: pieces of fp32 rows, aligned copies of bf16 rows, feature-major copies of
//                   activations for the structured-sparse path and the CUDA-core kernels (same rule).
//   MST_WS_ATTENTION  per-row dot products of the attention backward pass (same rule).
//   MST_WS_IMAGE    dense image of W.M (bf16, or the three pieces) of the layer being multiplied, for layers without
//                   value tracking (same rule).
mst_status_t mst_workspace_kind(int kind, size_t bytes, void** ptr) {
  constexpr int MAX_DEVICES = 64;
  static void* buf[MST_WS_KINDS][MAX_DEVICES] = {};
  static size_t cap[MST_WS_KINDS][MAX_DEVICES] = {};
  int dev = 0;
  MST_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= MAX_DEVICES || kind < 0 || kind >= MST_WS_KINDS) return MST_ERR_CUDA;
  if (bytes > cap[kind][dev]) {
    if (buf[kind][dev]) {
      MST_CUDA_TRY(cudaDeviceSynchronize());
      MST_CUDA_TRY(cudaFree(buf[kind][dev]));
      buf[kind][dev] = nullptr;
      cap[kind][dev] = 0;
    }
    const size_t want = (bytes + ((size_t)1 << 20)) & ~(((size_t)1 << 20) - 1);
    const cudaError_t got = cudaMalloc(&buf[kind][dev], want);
    if (got != cudaSuccess) cudaGetLastError();   // reported by the status: a later call must not find it again
    MST_CUDA_TRY(got);
    cap[kind][dev] = want;
  }
  *ptr = buf[kind][dev];
  return MST_OK;
}
mst_status_t mst_workspace(size_t bytes, void** ptr) { return mst_workspace_kind(MST_WS_SPLIT, bytes, ptr); }

bool mst_tc_gemm_usable(const void* A, int64_t lda, const void* B, int64_t ldb) {
  return (lda % 8 == 0) && (ldb % 8 == 0) && ((reinterpret_cast<uintptr_t>(A) & 15u) == 0) &&
         ((reinterpret_cast<uintptr_t>(B) & 15u) == 0) && mst_encode_tiled() != nullptr;
}

mst_tc_choice mst_tc_choose(const mst_tc_gemm_args& a) {
  mst_tc_choice c = {false, mst_env_any(), 0.0, {0, 0, 0.0}};
  // Few tiles: compare one wave of this kernel with the small-tile kernel's estimate, in SM clocks as there: a launch, the k-blocks of
  // a pair's tile, an epilogue that nothing overlaps in a single wave, and a second launch that adds the ranges and moves their sums.
  // Fitted to layers drawn over 96..4096 features (at most 4096 x 2048), or a block's of width 320..1280, and 17..4096 tokens, both kernels timed,
  // once for sizes of whole 16-byte pieces and once for odd ones, whose rows leave one by one and whose entries end in partial words and
  // squares.  Products: 190 layers, figures of the calls whose operands need no copies (3 to 8 % off the measured times, 7 to 33 before); activations
  // of odd rows, which travel 32 neighbours at a time: 169 and 168 calls, 1.1 and 1.9 % above the best of each (2.3 and 2.1 with the figures from before
  // they did); the derivative in one token tile 3.5 % above it (5.8 with 12900 + 603 a k-block).  Gradients: 511 layers, d = 0.02..0.5, with everything a call launches: where the entries do not leave with the contraction
  // or its sums, a sweep over the finished matrix follows.  Above the best kernel and number of ranges of each call, even / odd: entries 0.6 / 1.4 %, dense
  // 0.4 / 1.1, dense with entries 0.7 / 1.2; 1.1 / 1.4, 2.7 / 1.5 and 3.2 / 1.9 with the sweep left out and 148 blocks in clusters of any size
  // (2304 x 768, 1817 tokens, dense with entries: 18.7 us here, 14.3 in small tiles).
  if (!mst_getenv(c.env, "MST_TC_PAIR") && !mst_getenv(c.env, "MST_TC_SPLITS") && a.splits <= 1) {
    const int64_t tiles = ((a.M + 2 * BM - 1) / (2 * BM)) * ((a.N + BN - 1) / BN), kb = (a.K + BK - 1) / BK, pairs = mst_sm_count() / 2;
    if (tiles <= pairs) {
      double here;
      if (a.epilogue == MST_TC_OUT_BF16) {
        const bool even = a.ldc % 8 == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0 &&
                          (!a.act || !a.pre || (a.ldpre % 8 == 0 && (reinterpret_cast<uintptr_t>(a.pre) & 15u) == 0));
        const double k = (double)kb;
        const bool grad = a.act == MST_ACT_GELU_GRAD;
        if (!a.act) here = a.M <= BM ? 8350.0 + k * 606.0 : even ? 8350.0 + k * 460.0 : 10400.0 + k * 552.0;   // one token tile: single blocks
        else if (a.M <= BM) here = even ? (grad ? 16000.0 + k * 500.0 : 12900.0 + k * 603.0) : grad ? 26500.0 + k * 570.0 : 20000.0 + k * 579.0;
        else if (even) here = grad ? 10800.0 + k * 462.0 : 10750.0 + k * 478.0;
        else here = (grad ? 17000.0 + k * 450.0 : 13600.0 + k * 560.0) + (grad ? 0.0030 : 0.0025) * (double)a.M * (double)a.N;
      } else {
        const bool entries = a.epilogue == MST_TC_OUT_SAMPLED, even = a.M % 8 == 0 && a.N % 8 == 0;
        const double out_bytes = entries ? 4.0 * (double)a.nnz : 4.0 * (double)a.M * (double)a.N;
        int cut;
        const int64_t sp = mst_tc_pick_splits(tiles, pairs, kb, out_bytes, &cut), per = (kb + sp - 1) / sp;
        // the entries come with the sums of several ranges, or from the finished matrix
        const bool sweep = a.also_sampled && !(a.M > BM && sp > 1 && a.N % 4 == 0);
        if (entries) {
          const bool few = (double)a.nnz * 1024.0 < SAMPLED_STAGE_MIN * (double)a.M * (double)a.N;
          here = even ? (few ? 10500.0 : 12900.0) + (double)per * 588.0 : (few ? 12000.0 : 14000.0) + (double)per * 574.0;
          if (sp > 1) here += even ? 3330.0 + (double)sp * out_bytes * 1.17e-3 : 3500.0 + (double)sp * out_bytes * 7.4e-4;   // written and read
        } else if (even) {
          here = a.also_sampled ? 13900.0 + (double)per * 548.0 + (sweep ? 4780.0 : 0.0) : 11500.0 + (double)per * 568.0;
          if (sp > 1) here += (a.also_sampled ? -150.0 : 2020.0) + (double)sp * out_bytes * (a.also_sampled ? 5.1e-4 : 4.0e-4);
        } else {
          here = 17100.0 + (double)per * 510.0 + (sp > 1 ? 5700.0 : 0.0) + (sweep ? 5000.0 : 0.0);
        }
      }
      c.plan = mst_tc_small_plan(a);
      c.small = c.plan.clocks < here;
      c.clocks = c.small ? c.plan.clocks : here;
    }
  }
  return c;
}

mst_status_t mst_tc_gemm(const mst_tc_gemm_args& a, const mst_tc_choice& choice, cudaStream_t s) {
  if (a.M <= 0 || a.N <= 0 || a.K <= 0) return MST_ERR_INVALID_ARG;
  if (!mst_tc_gemm_usable(a.A, a.lda, a.B, a.ldb)) return MST_ERR_SHAPE;
  if (choice.small) return mst_tc_small(a, choice.plan, s);
  const bool env = choice.env;
  CUtensorMap tmA, tmB;
  // Block pairs (256-row tiles) pay off once there are at least two row tiles; MST_TC_PAIR=0/1 overrides.
  bool pair = a.M > BM;
  if (const char* e = mst_getenv(env, "MST_TC_PAIR")) pair = (e[0] == '1');
  // K-major: [rows x K], box 64 (K) x tile rows.  MN-major: [K x rows], box 64 (rows) x BK.
  const bool okA = a.a_mn_major ? make_map(&tmA, a.A, a.K, a.M, a.lda, BK) : make_map(&tmA, a.A, a.M, a.K, a.lda, BM);
  const int b_rows = pair ? BN / 2 : BN;
  const bool okB = a.b_mn_major ? make_map(&tmB, a.B, a.K, a.N, a.ldb, BK) : make_map(&tmB, a.B, a.N, a.K, a.ldb, b_rows);
  if (!okA || !okB) return MST_ERR_SHAPE;
  Params P;
  P.M = a.M;
  P.N = a.N;
  P.kblocks = (int)((a.K + BK - 1) / BK);
  P.splits = 1;
  P.cut = 1;
  int sums = 1;   // partial sums kept for one output at most
  P.m_tiles = (int)((a.M + BM - 1) / BM);
  P.n_tiles = (int)((a.N + BN - 1) / BN);
  P.epilogue = a.epilogue;
  P.major = a.a_mn_major ? M_GRADIENT : a.b_mn_major ? M_INPUT : M_FORWARD;
  P.out = a.out;
  P.ldc = a.ldc;
  P.partial = nullptr;
  P.bits = a.bits;
  P.wscan = a.wscan;
  P.wpr = a.wpr;
  P.nnz = a.nnz;
  P.act = a.epilogue == MST_TC_OUT_BF16 ? a.act : 0;
  P.pre = a.pre;
  P.ldpre = a.ldpre;
  P.redo = a.redo;
  if (P.act == MST_ACT_GELU_GRAD && !P.pre) return MST_ERR_INVALID_ARG;
  P.sampled_stage_min = SAMPLED_STAGE_MIN;
  if (const char* e = mst_getenv(env, "MST_TC_SAMPLED_STAGE")) P.sampled_stage_min = atoi(e);  // measurement override
  if (a.epilogue != MST_TC_OUT_BF16) {
    // few output tiles: cut the contraction range so that all SMs work; partial sums go to the shared scratch buffer
    const int64_t works1 = pair ? (int64_t)((P.m_tiles + 1) / 2) * P.n_tiles : (int64_t)P.m_tiles * P.n_tiles;
    const int64_t slots = pair ? mst_sm_count() / 2 : mst_sm_count();
    const double out_bytes = a.epilogue == MST_TC_OUT_F32 ? 4.0 * (double)a.M * (double)a.N : 4.0 * (double)a.nnz;
    int cut = 1;
    P.splits = a.splits > 0 ? a.splits : mst_tc_pick_splits(works1, slots, P.kblocks, out_bytes, &cut);
    if (const char* e = mst_getenv(env, "MST_TC_SPLITS")) {  // measurement override
      const int v = atoi(e);
      if (v > 0) { P.splits = v; cut = 1; }
    }
    if (P.splits > P.kblocks) P.splits = P.kblocks;
    if (pair) P.cut = (uint32_t)cut;
    sums = P.splits + (int)P.cut - 1;
    if (sums > 1) {
      const size_t per = a.epilogue == MST_TC_OUT_F32 ? (size_t)a.M * a.N : (size_t)a.nnz;
      void* ws = nullptr;
      MST_TRY(mst_workspace(sizeof(float) * per * sums, &ws));
      P.partial = (float*)ws;
    }
  }
  // staged epilogue when the output (and the pre-activation) can be described to the TMA unit (MST_TC_TMA_OUT=0 keeps per-thread stores)
  CUtensorMap tmC = tmA, tmP = tmA;
  bool tma_out = false;
  P.whole = (int)a.N & ~7;
  if (a.epilogue == MST_TC_OUT_BF16) {
    // pre-activations that are read may end anywhere
    tma_out = P.whole > 0 && make_out_map_bf16(&tmC, a.out, a.M, P.whole, a.ldc) &&
              (!P.act || !P.pre || make_out_map_bf16(&tmP, P.pre, a.M, P.act == MST_ACT_GELU ? P.whole : a.N, P.ldpre));
  } else if (a.epilogue == MST_TC_OUT_F32) {
    tma_out = a.N % 4 == 0 && (sums > 1 ? make_out_map_f32(&tmC, P.partial, a.M, a.N, a.N, a.M * a.N, sums)
                                        : make_out_map_f32(&tmC, a.out, a.M, a.N, a.ldc, a.M * a.ldc, 1));
  }
  if (const char* e = mst_getenv(env, "MST_TC_TMA_OUT")) {
    if (e[0] == '0') tma_out = false;
  }
  const int kind = a.epilogue == MST_TC_OUT_SAMPLED ? K_SAMPLED : !tma_out ? (P.act ? K_ROWS_ACT : K_ROWS) : 
                   a.epilogue == MST_TC_OUT_F32 ? K_F32 : P.redo.kind || P.whole != a.N ? (P.act ? K_REDO_ACT : K_REDO) : P.act ? K_ACT : K_BF16;
  if (pair) {
    const int64_t jobs = (int64_t)((P.m_tiles + 1) / 2) * P.n_tiles * P.splits, max_pairs = mst_sm_count() / 2, rest = jobs % max_pairs;
    CUtensorMap tmBn = tmB;
    if (a.epilogue == MST_TC_OUT_BF16) {
      // half-wide tiles take about 0.62 of a full one (at most twice as many blocks share the L2 bandwidth that bounds them)
      if (rest * 2 <= max_pairs) P.cut = 2;
      if (!a.b_mn_major && !make_map(&tmBn, a.B, a.N, a.K, a.ldb, BN / 4)) return MST_ERR_SHAPE;
    }
    P.full = (uint32_t)(P.cut > 1 ? jobs - rest : jobs);
    const int64_t works = (int64_t)P.full + (int64_t)P.cut * (jobs - (int64_t)P.full);
    if (works > 0x7FFFFFFF) return MST_ERR_SHAPE;
    const dim3 grid(2 * (unsigned)(works < max_pairs ? works : max_pairs));
#define MST_LAUNCH_KIND(K, M)                                                                                         \
  case 8 * M + K:                                                                                                     \
    MST_SMEM_LIMIT((tc_gemm_pair_kernel<K, M>), P_SMEM_BYTES);                                                        \
    MST_CUDA_TRY(mst_launch_overlapped(tc_gemm_pair_kernel<K, M>, grid, dim3(NUM_THREADS), P_SMEM_BYTES, s, tmA, tmB, tmBn, tmC, tmP, P)); \
    break
    switch (8 * P.major + kind) {
      MST_LAUNCH_KIND(K_BF16, M_FORWARD);
      MST_LAUNCH_KIND(K_ACT, M_FORWARD);
      MST_LAUNCH_KIND(K_REDO, M_FORWARD);
      MST_LAUNCH_KIND(K_REDO_ACT, M_FORWARD);
      MST_LAUNCH_KIND(K_ROWS, M_FORWARD);
      MST_LAUNCH_KIND(K_ROWS_ACT, M_FORWARD);
      MST_LAUNCH_KIND(K_BF16, M_INPUT);
      MST_LAUNCH_KIND(K_ACT, M_INPUT);
      MST_LAUNCH_KIND(K_REDO, M_INPUT);
      MST_LAUNCH_KIND(K_REDO_ACT, M_INPUT);
      MST_LAUNCH_KIND(K_ROWS, M_INPUT);
      MST_LAUNCH_KIND(K_ROWS_ACT, M_INPUT);
      MST_LAUNCH_KIND(K_F32, M_GRADIENT);
      MST_LAUNCH_KIND(K_SAMPLED, M_GRADIENT);
      MST_LAUNCH_KIND(K_ROWS, M_GRADIENT);
      default: return MST_ERR_INVALID_ARG;
    }
#undef MST_LAUNCH_KIND
  } else {
    const int64_t works = (int64_t)P.m_tiles * P.n_tiles * P.splits;
    const int grid = (int)(works < mst_sm_count() ? works : mst_sm_count());
#define MST_LAUNCH_KIND(K)                                                                                            \
  case K:                                                                                                             \
    MST_SMEM_LIMIT((tc_gemm_kernel<K>), SMEM_BYTES);                                                                  \
    MST_CUDA_TRY(mst_launch_overlapped(tc_gemm_kernel<K>, dim3(grid), dim3(NUM_THREADS), SMEM_BYTES, s, tmA, tmB, tmC, tmP, P)); \
    break
    switch (kind) {
      MST_LAUNCH_KIND(K_BF16);
      MST_LAUNCH_KIND(K_F32);
      MST_LAUNCH_KIND(K_SAMPLED);
      MST_LAUNCH_KIND(K_ACT);
      MST_LAUNCH_KIND(K_REDO);
      MST_LAUNCH_KIND(K_REDO_ACT);
      MST_LAUNCH_KIND(K_ROWS);
      MST_LAUNCH_KIND(K_ROWS_ACT);
    }
#undef MST_LAUNCH_KIND
  }
  MST_CUDA_TRY(cudaGetLastError());
  if (a.also_sampled && pair && sums > 1 && a.epilogue == MST_TC_OUT_F32 && a.N % 4 == 0 && a.ldc % 4 == 0 &&
      (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0) {
    MST_CUDA_TRY(mst_launch_overlapped(tc_reduce_sample_kernel, dim3((unsigned)((P.M + 7) / 8), (unsigned)((P.N + 127) / 128)), dim3(256), 0, s, P,
                                       a.also_sampled));
    *a.sampled = true;
  } else if (pair && P.cut > 1 && sums > 1) {
    MST_CUDA_TRY(mst_launch_overlapped(tc_reduce_tiles_kernel, dim3((unsigned)((P.M + 7) / 8), (unsigned)P.n_tiles), dim3(256), 0, s, P));
  } else if (P.splits > 1) {
    const int64_t n = a.epilogue == MST_TC_OUT_F32 ? a.M * a.N : a.nnz;
    if (n > 0 && (n & 3) == 0 && (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0)
      MST_CUDA_TRY(mst_launch_overlapped(tc_reduce4_kernel, dim3((unsigned)((n / 4 + 255) / 256)), dim3(256), 0, s,
                                         (const float4*)P.partial, P.splits, n / 4, (float4*)a.out));
    else if (n > 0)
      MST_CUDA_TRY(mst_launch_overlapped(tc_reduce_kernel, dim3((unsigned)((n + 255) / 256)), dim3(256), 0, s,
                                         (const float*)P.partial, P.splits, n, (float*)a.out));
    MST_CUDA_TRY(cudaGetLastError());
  }
  return MST_OK;
}

extern "C" mst_status_t mst_device_error_flags(int32_t* flags) {
  if (!flags) return MST_ERR_INVALID_ARG;
  int v = 0;
  MST_CUDA_TRY(cudaDeviceSynchronize());
  MST_CUDA_TRY(cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int)));
  int32_t att = 0;
  MST_TRY(mst_attention_error_flags(&att));
  int32_t sp = 0, cc = 0;
  MST_TRY(mst_sp24_error_flags(&sp));
  MST_TRY(mst_spmm_error_flags(&cc));
  int32_t sd = 0;
  MST_TRY(mst_sddmm_error_flags(&sd));
  cc |= sd;
  int32_t f32 = 0;
  MST_TRY(mst_split_error_flags(&f32));
  v |= f32;
  *flags = v | (att << 1) | (sp << 2) | (cc << 3);
  return MST_OK;
}
