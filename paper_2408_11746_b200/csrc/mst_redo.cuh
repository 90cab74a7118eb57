// Results that a product over dense pieces cannot give, formed again from the operands as the caller has them.
//
// A product over stored entries leaves alone what it does not store: an infinite or NaN activation reaches the outputs connected to
// it and no others.  The dense image multiplies it by every masked zero, and a value cut into bf16 pieces by the zero pieces of its
// partner, so that one such value made a NaN of every output of its row.  fp32 calls and bf16 calls on rows the TMA unit does not
// take (the calls that have always gone over stored entries) therefore look at their sums on the way out: a sum that is not finite
// is formed again, term by term in fp32, over the stored entries (products) or over the tokens (gradients).  Sums that are finite
// had only finite terms and are left as they are.
// The test is one multiply-add per sum by the thread that holds it (2051 x 1023 bf16 at 1999 tokens, all three
// products: 57.1 -> 57.9 us; 3072 x 768 fp32 step at 256 tokens, with the scaled pieces: 131.8 -> 135.0).  What follows a find is for
// runs that have gone wrong and is slower than the CUDA-core kernels (one warp per 32 x 32 square, from global memory): forward of the
// 3072 x 768 fp32 layer at 256 tokens 0.40 ms with one infinite activation and 0.47 with all NaN (CUDA cores 0.08), of a 769 x 3073 bf16
// layer at 8192 tokens 3.7 and 7.8 ms (0.57); column by column it was 1.1 and 1.8, 10.6 and 57 ms.  Operands in flight: four of each; eight
// left the contraction kernels' epilogues with spilled registers, 2 % of the fused activation.
#pragma once
#include <stdint.h>

#include "mst_tc_gemm.cuh"

__device__ __forceinline__ float mst_redo_f32(float v) { return v; }
__device__ __forceinline__ float mst_redo_f32(uint16_t v) { return __uint_as_float((uint32_t)v << 16); }

// sum * 0 over finite values is 0, otherwise NaN
__device__ __forceinline__ bool mst_redo_needed(float v) { return !(v * 0.f == 0.f); }

// One warp, converged: v[0..31] = columns n .. n + 31 of row `row` (rows: lane 0's .. lane 31's), mine = this lane has a row.
// Values that are not finite are replaced.
template <typename V>
static __device__ __noinline__ void mst_redo_square(const mst_redo R, float* v, int64_t row, bool mine, int64_t n, int64_t N) {
  const int lane = threadIdx.x & 31;
  if (R.kind == MST_REDO_GRADIENT) {
    // loads are never conditional (lanes without a row or column read the first, tokens past the last repeat it): four of each fly together
    const bool col = n + lane < N;
    const V* A = (const V*)R.A + (mine ? row : 0);
    const V* B = (const V*)R.B + (col ? n + lane : 0);
    float acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
#pragma unroll 1
    for (int64_t t0 = 0; t0 < R.K; t0 += 4) {
      V a[4], b[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t t = t0 + u < R.K ? t0 + u : R.K - 1;
        a[u] = A[t * R.lda];
        b[u] = B[t * R.ldb];
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const bool in = t0 + u < R.K;                               // otherwise 0 * 0
        const float av = in ? mst_redo_f32(a[u]) : 0.f, bv = in ? mst_redo_f32(b[u]) : 0.f;
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = fmaf(av, __shfl_sync(0xffffffffu, bv, j), acc[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (mine && mst_redo_needed(v[j])) v[j] = acc[j];
    return;
  }
  const V* A = (const V*)R.A + (mine ? row : 0) * R.lda;
  const V* vals = (const V*)R.B;
  const bool forward = R.kind == MST_REDO_FORWARD;
  float acc[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) acc[j] = 0.f;
  for (int64_t k0 = 0; k0 < R.K; k0 += 32) {
    const int count = R.K - k0 < 32 ? (int)(R.K - k0) : 32;
    // forward: a lane keeps its column's mask word over these contraction indices; input gradient: a lane keeps an index's word
    // over the columns (n is a multiple of 32)
    const int64_t o = forward ? n + lane : k0 + lane, wi = o * R.wpr + ((forward ? k0 : n) >> 5);
    uint32_t word = 0;
    int32_t first = 0;
    if (forward ? o < N : lane < count) {
      word = R.bits[wi];
      first = R.wscan[wi];
    }
#pragma unroll 1
    for (int e0 = 0; e0 < count; e0 += 4) {
      V w[4], x[4];
      uint32_t stored = 0;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int e = e0 + u;                                       // at most 31: beyond `count` nothing is stored
        const uint32_t mask = forward ? word : __shfl_sync(0xffffffffu, word, e);
        const int32_t at = forward ? first : __shfl_sync(0xffffffffu, first, e);
        const int bit = forward ? e : lane;
        const bool has = (mask >> bit) & 1u;                        // (index k0 + e, column n + lane) is stored
        w[u] = vals[has ? at + __popc(mask & ((1u << bit) - 1u)) : 0];
        x[u] = A[k0 + (e < count ? e : 0)];
        stored |= has ? 1u << u : 0u;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const uint32_t columns = __ballot_sync(0xffffffffu, (stored >> u) & 1u);
        const float wv = mst_redo_f32(w[u]), xv = mst_redo_f32(x[u]);
#pragma unroll
        for (int j = 0; j < 32; ++j) {
          const float sum = fmaf(__shfl_sync(0xffffffffu, wv, j), xv, acc[j]);
          acc[j] = (columns >> j) & 1u ? sum : acc[j];
        }
      }
    }
  }
#pragma unroll
  for (int j = 0; j < 32; ++j)
    if (mine && n + j < N && mst_redo_needed(v[j])) v[j] = acc[j];
}

// One thread: one output of a forward product
template <typename V>
static __device__ __noinline__ float mst_redo_one(const mst_redo R, int64_t row, int64_t c) {
  const V* A = (const V*)R.A + row * R.lda;
  const V* vals = (const V*)R.B;
  float acc = 0.f;
  for (int wc = 0; wc < R.wpr; ++wc) {
    int32_t at = R.wscan[c * R.wpr + wc];
    for (uint32_t word = R.bits[c * R.wpr + wc]; word; word &= word - 1u)
      acc = fmaf(mst_redo_f32(vals[at++]), mst_redo_f32(A[wc * 32 + __ffs(word) - 1]), acc);
  }
  return acc;
}
