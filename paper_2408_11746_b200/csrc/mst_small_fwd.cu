// Forward product for a few tokens (sampling, tiny batches):  Y[t, o] = sum_k X[t, k] * image[o, k],  image = W.M in bf16.
//
// What bounds it: latency.  The image is read once (14 MB for a GPT-2-small block, from L2 when it is reused) and the sums are
// a few million, so the time is one launch plus one round trip to memory, if enough loads are in flight.  A 128 x 256 tcgen05
// tile leaves 139 of 148 SMs idle here and walks through the contraction range one block after the other (11-19 us per layer).
// Instead a block takes 16 output features and all of its warps share their contraction range, 32 indices at a
// time; fragments go from global memory straight to registers: the order of the contraction indices is free as long as both
// operands agree, so a lane's eight neighbouring values (one 16-byte load) serve as the k-pairs of two m16n8k16 products.  The
// warps' sums meet in shared memory in a fixed order.  Measured at 16 tokens: 3-4 us per layer of a GPT-2-small block.
#include "mst_internal.cuh"
#include "mst_redo.cuh"
#include "mst_tc_gemm.cuh"

#include <cuda_bf16.h>

namespace {

__device__ __forceinline__ void mma_bf16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, {%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

// NT: groups of 8 tokens per block.  REDO: sums that are not finite are formed again (a kernel of its own: the call in the epilogue cost
// the four layers of a GPT-2-small block at 16 tokens 0.6 us)
template <int NT, int SF_WARPS, bool REDO>
__global__ void __launch_bounds__(32 * SF_WARPS)
small_fwd_kernel(const uint16_t* __restrict__ X, int64_t ldx, int T, const uint16_t* __restrict__ W, int64_t ldw, int O, int K,
                 __nv_bfloat16* __restrict__ Y, int64_t ldy, int act, __nv_bfloat16* __restrict__ pre, int64_t ldpre, const mst_redo redo) {
  __shared__ float red[SF_WARPS][NT * 8][17];
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int o0 = blockIdx.x * 16, t0 = blockIdx.y * NT * 8;
  float acc[NT][4];
#pragma unroll
  for (int n = 0; n < NT; ++n)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[n][j] = 0.f;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  const bool r0 = o0 + g < O, r1 = o0 + g + 8 < O;
  const uint16_t* w0 = W + (int64_t)(r0 ? o0 + g : 0) * ldw + t * 8;
  const uint16_t* w1 = W + (int64_t)(r1 ? o0 + g + 8 : 0) * ldw + t * 8;
  const int chunks = (K + 31) / 32;
  constexpr int U = 4;   // chunks in flight
  for (int c0 = warp; c0 < chunks; c0 += SF_WARPS * U) {
    uint4 a0[U], a1[U], b[U][NT];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k = (c0 + u * SF_WARPS) * 32;
      const bool in = k + t * 8 < K;   // the rows are padded with zeros to a multiple of 8
      a0[u] = in && r0 ? __ldg(reinterpret_cast<const uint4*>(w0 + k)) : zero;
      a1[u] = in && r1 ? __ldg(reinterpret_cast<const uint4*>(w1 + k)) : zero;
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        const int tok = t0 + n * 8 + g;
        b[u][n] = in && tok < T ? __ldg(reinterpret_cast<const uint4*>(X + (int64_t)tok * ldx + k + t * 8)) : zero;
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int n = 0; n < NT; ++n) {
        mma_bf16(acc[n], a0[u].x, a1[u].x, a0[u].y, a1[u].y, b[u][n].x, b[u][n].y);
        mma_bf16(acc[n], a0[u].z, a1[u].z, a0[u].w, a1[u].w, b[u][n].z, b[u][n].w);
      }
  }
#pragma unroll
  for (int n = 0; n < NT; ++n) {
    red[warp][n * 8 + 2 * t][g] = acc[n][0];
    red[warp][n * 8 + 2 * t + 1][g] = acc[n][1];
    red[warp][n * 8 + 2 * t][g + 8] = acc[n][2];
    red[warp][n * 8 + 2 * t + 1][g + 8] = acc[n][3];
  }
  __syncthreads();
  for (int i = threadIdx.x; i < NT * 8 * 16; i += 32 * SF_WARPS) {
    const int f = i & 15, n = i >> 4, o = o0 + f, tok = t0 + n;
    if (o >= O || tok >= T) continue;
    float v = red[0][n][f];
#pragma unroll
    for (int w = 1; w < SF_WARPS; ++w) v += red[w][n][f];
    if (REDO && mst_redo_needed(v)) v = mst_redo_one<uint16_t>(redo, tok, o);
    if (act == MST_ACT_GELU) {
      if (pre) pre[(int64_t)tok * ldpre + o] = __float2bfloat16_rn(v);
      v = mst_gelu(v);
    }
    Y[(int64_t)tok * ldy + o] = __float2bfloat16_rn(v);
  }
}

template <int NT, int SF_WARPS>
mst_status_t launch_warps(const void* X, int64_t ldx, int64_t T, const uint16_t* image, int64_t ldimage, int O, int K, void* Y, int64_t ldy,
                          int act, void* pre, int64_t ldpre, const mst_redo& redo, cudaStream_t s) {
  MST_CUDA_TRY(mst_launch_overlapped(redo.kind ? small_fwd_kernel<NT, SF_WARPS, true> : small_fwd_kernel<NT, SF_WARPS, false>, dim3((unsigned)((O + 15) / 16), (unsigned)((T + NT * 8 - 1) / (NT * 8))),
                                     dim3(32 * SF_WARPS), 0, s, (const uint16_t*)X, ldx, (int)T, image, ldimage, O, K, (__nv_bfloat16*)Y,
                                     ldy, act, (__nv_bfloat16*)pre, ldpre, redo));
  return MST_OK;
}

// As many warps as give each four chunks of the range, one trip to memory (768 x 3072: 5.8 us with 8 warps and three trips, 4.4 with 24)
template <int NT>
mst_status_t launch_small(const void* X, int64_t ldx, int64_t T, const uint16_t* image, int64_t ldimage, int O, int K, void* Y, int64_t ldy,
                          int act, void* pre, int64_t ldpre, const mst_redo& redo, cudaStream_t s) {
  if (K <= 1024) return launch_warps<NT, 8>(X, ldx, T, image, ldimage, O, K, Y, ldy, act, pre, ldpre, redo, s);
  if (K <= 2048) return launch_warps<NT, 16>(X, ldx, T, image, ldimage, O, K, Y, ldy, act, pre, ldpre, redo, s);
  return launch_warps<NT, 24>(X, ldx, T, image, ldimage, O, K, Y, ldy, act, pre, ldpre, redo, s);
}

}  // namespace

// A launch with its trip to memory, and the 64 K bytes that each block of 16 tokens and 16 features reads, at what L2 delivers to all SMs, with
// what a block costs beside them; figures for each number of warps (launch_small).  Fitted to 212 forward calls without copies, drawn over
// 96..5120 features and 17..1024 tokens, 5 to 9 % off their times; one figure for all (15 % off) had 717 x 114 -> 3712 take 33 us here
// instead of 10 in small tiles.  Small tiles from 17 tokens on, as they once were: 42 % above the better kernel (a GPT-2-small block
// at 17, 32, 64 tokens: 29.6 -> 16.3 us, 30.3 -> 16.1, 30.4 -> 23.0; at GPT-2-large width and 64 tokens the tiles win, 40 against 50).
double mst_small_fwd_clocks(int64_t T, int O, int K) {
  const double bytes = (double)((O + 15) / 16) * (double)((T + 15) / 16) * 64.0;   // per index of the contraction range
  if (K <= 1024) return 6200.0 + bytes * (double)(K + 404) / 8980.0;
  if (K <= 2048) return 5700.0 + bytes * (double)(K + 3060) / 16330.0;
  return 5500.0 + bytes * (double)(K + 1040) / 5600.0;
}

// X rows 16-byte aligned, columns K .. multiple of 8 zero in X and in the image; act NONE or GELU
mst_status_t mst_small_fwd(const void* X, int64_t ldx, int64_t T, const uint16_t* image, int64_t ldimage, int O, int K, void* Y, int64_t ldy,
                           int act, void* pre, int64_t ldpre, const mst_redo& redo, cudaStream_t s) {
  if (T <= 8) return launch_small<1>(X, ldx, T, image, ldimage, O, K, Y, ldy, act, pre, ldpre, redo, s);
  return launch_small<2>(X, ldx, T, image, ldimage, O, K, Y, ldy, act, pre, ldpre, redo, s);
}
