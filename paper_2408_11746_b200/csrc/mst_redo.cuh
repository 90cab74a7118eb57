// Results that a product over dense pieces cannot give, formed again from the operands as the caller has them.
//
// A product over stored entries leaves alone what it does not store: an infinite or NaN activation reaches the outputs connected to
// it and no others.  The dense image multiplies it by every masked zero, and a value cut into bf16 pieces by the zero pieces of its
// partner, so that one such value made a NaN of every output of its row.  fp32 calls and bf16 calls on rows the TMA unit does not
// take (the calls that have always gone over stored entries) therefore look at their sums on the way out: a sum that is not finite
// is formed again, term by term in fp32, over the stored entries (products) or over the tokens (gradients).  Sums that are finite
// had only finite terms and are left as they are.
// The test is one multiply-add per sum by the thread that holds it (2051 x 1023 bf16 at 1999 tokens, all three
// products: 57.1 -> 57.9 us; 3072 x 768 fp32 step at 256 tokens, with the scaled pieces: 131.8 -> 135.0).  What follows a find is far slower than the tensor cores (one
// warp per 32 x 32 square, from global memory) and bounded by the work of the CUDA-core kernels times a small factor.
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
    const V* A = (const V*)R.A + row;
    const V* B = (const V*)R.B + n + lane;
    const bool col = n + lane < N;
    float acc[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) acc[j] = 0.f;
    for (int64_t t = 0; t < R.K; ++t) {
      const float a = mine ? mst_redo_f32(A[t * R.lda]) : 0.f, b = col ? mst_redo_f32(B[t * R.ldb]) : 0.f;
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[j] = fmaf(a, __shfl_sync(0xffffffffu, b, j), acc[j]);
    }
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (mine && mst_redo_needed(v[j])) v[j] = acc[j];
    return;
  }
  const V* A = (const V*)R.A + row * R.lda;
  const V* vals = (const V*)R.B;
  for (int j = 0; j < 32 && n + j < N; ++j) {
    const int64_t c = n + j;
    const bool need = mine && mst_redo_needed(v[j]);
    if (!__any_sync(0xffffffffu, need)) continue;
    float acc = 0.f;
    for (int64_t k0 = 0; k0 < R.K; k0 += 32) {
      // a lane per contraction index: is (row, column) of the weight stored, and where
      const int64_t k = k0 + lane;
      const int64_t o = R.kind == MST_REDO_FORWARD ? c : k, i = R.kind == MST_REDO_FORWARD ? k : c;
      float w = 0.f;
      bool has = false;
      if (k < R.K) {
        const uint32_t word = R.bits[o * R.wpr + (i >> 5)], below = (1u << (i & 31)) - 1u;
        has = (word >> (i & 31)) & 1u;
        if (has) w = mst_redo_f32(vals[R.wscan[o * R.wpr + (i >> 5)] + __popc(word & below)]);
      }
      const uint32_t m = __ballot_sync(0xffffffffu, has);
#pragma unroll
      for (int g = 0; g < 32; g += 8) {
        if (!((m >> g) & 0xFFu)) continue;   // uniform
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          x[e] = 0.f;
          if (need && ((m >> (g + e)) & 1u)) x[e] = mst_redo_f32(A[k0 + g + e]);
        }
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const float ww = __shfl_sync(0xffffffffu, w, g + e);
          if ((m >> (g + e)) & 1u) acc = fmaf(ww, x[e], acc);
        }
      }
    }
    if (need) v[j] = acc;
  }
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
