// Interface of the tcgen05 (5th-generation tensor core) bf16 contraction used for the dense gradient,
// the dense-tile SpMM path and the sampled weight gradient.  Internal to libmst.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mst.h"

// C[M x N] = A * B^T-like contraction over K with fp32 accumulation in tensor memory.
//   A operand: K-major   -> A is stored [M x K] row-major (lda elements between rows), or
//              MN-major  -> A is stored [K x M] row-major (lda elements between K rows)
//   B operand: K-major   -> B is stored [N x K] row-major, or MN-major -> [K x N] row-major
// Epilogues:
//   MST_TC_OUT_BF16     C bf16 row-major [M x ldc]
//   MST_TC_OUT_F32      C fp32 row-major [M x ldc]; with splits > 1 writes partial sums to
//                       partial[split][M x N] (contiguous) which mst_tc_reduce then sums in a fixed order
//   MST_TC_OUT_SAMPLED  only entries under a bit mask are written, to their CSR position:
//                       out[wscan[w] + rank] for mask word w = m*wpr + n/32 (needs N-tile offsets multiple of 32)
enum { MST_TC_OUT_BF16 = 0, MST_TC_OUT_F32 = 1, MST_TC_OUT_SAMPLED = 2 };

// Element-wise step fused into the bf16 epilogue (GPT-2 MLP: fc1 -> GELU -> fc2, erf form):
//   GELU       out = gelu(acc), optionally pre = acc
//   GELU_GRAD  out = acc * gelu'(pre)
enum { MST_ACT_NONE = 0, MST_ACT_GELU = 1, MST_ACT_GELU_GRAD = 2 };

__host__ __device__ inline float mst_gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__host__ __device__ inline float mst_gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// Operands from which sums that are not finite are formed again (mst_redo.cuh); kind 0: they stay
enum { MST_REDO_FORWARD = 1, MST_REDO_BACKWARD = 2, MST_REDO_GRADIENT = 3 };
struct mst_redo {
  int kind;
  int wpr;               // products: mask words per row, and the mask
  const uint32_t* bits;
  const int32_t* wscan;
  const void* A;         // products: activations [M x K]; gradient: dY [K x M]
  int64_t lda;
  const void* B;         // products: stored values; gradient: X [K x N]
  int64_t ldb;
  int64_t K;
};

struct mst_tc_gemm_args {
  const void* A;
  int64_t lda;
  int a_mn_major;
  const void* B;
  int64_t ldb;
  int b_mn_major;
  int64_t M, N, K;
  int epilogue;
  void* out;
  int64_t ldc;
  int splits;            // 0 = choose; otherwise K is cut into this many contiguous ranges (F32 / SAMPLED epilogues);
                         // partial sums live in the process-wide scratch buffer and are added in a fixed order
  const uint32_t* bits;  // SAMPLED: mask words, wpr per row
  const int32_t* wscan;  // SAMPLED: exclusive popcount scan of the words
  int wpr;
  int64_t nnz;           // SAMPLED: number of stored entries (partial stride)
  int act;               // BF16 epilogue only: MST_ACT_NONE / MST_ACT_GELU / MST_ACT_GELU_GRAD
  void* pre;             // GELU: optional bf16 output for the pre-activation (may be NULL);
                         // GELU_GRAD: bf16 input holding the pre-activation the derivative is taken at
  int64_t ldpre;
  float* also_sampled;   // F32: the entries under the mask (bits, wscan, wpr) as well, where partial sums are added up anyway or tiles are small;
  bool* sampled;         //      set to true when that was done
  mst_redo redo;         // BF16 epilogue and mst_tc_split: sums that are not finite are formed again
};

// C = A * B with fp32 accuracy from operands given as three bf16 pieces each (mst_prepare.cu; lda / ldb are the pieces'
// leading dimensions, M / N / K the matrix sizes).  Epilogues F32 (rows) and SAMPLED.
mst_status_t mst_tc_split(const mst_tc_gemm_args& a, cudaStream_t s);
// The same kernel for bf16 operands and outputs of few tiles, all epilogues: tile width and K ranges with their estimated time in SM clocks,
// and the call with them
struct mst_small_plan { int bn, splits; double clocks; };
mst_small_plan mst_tc_small_plan(const mst_tc_gemm_args& a);
mst_status_t mst_tc_small(const mst_tc_gemm_args& a, const mst_small_plan& plan, cudaStream_t s);
// forward product of a few tokens (mst_small_fwd.cu): always up to MST_SMALL_FWD_TOKENS, up to MST_SMALL_FWD_MOST where its estimated time,
// in SM clocks as above, is shorter than the small tiles'
constexpr int64_t MST_SMALL_FWD_TOKENS = 16, MST_SMALL_FWD_MOST = 1024;
double mst_small_fwd_clocks(int64_t T, int O, int K);
mst_status_t mst_small_fwd(const void* X, int64_t ldx, int64_t T, const uint16_t* image, int64_t ldimage, int O, int K, void* Y, int64_t ldy,
                           int act, void* pre, int64_t ldpre, const mst_redo& redo, cudaStream_t s);

// dY^T X over T tokens with the sizes and the epilogue in `a` (M = O, N = I, K = T; F32 or SAMPLED), operands as the caller
// has them (mst_dense_grad.cu)
mst_status_t mst_tc_gradient(mst_tc_gemm_args a, mst_dtype_t dtype, const void* dY, int64_t lddy, const void* X, int64_t ldx,
                             cudaStream_t s);

// Returns MST_ERR_SHAPE when the operands cannot be described to the TMA unit (leading dimension or base address
// not 16-byte aligned); callers pass aligned copies of such rows (mst_prepare).
// The choice of its kernel is made once a call; `clocks` is the chosen one's estimate where one was made, else 0.
struct mst_tc_choice { bool small, env; double clocks; mst_small_plan plan; };
mst_tc_choice mst_tc_choose(const mst_tc_gemm_args& a);
mst_status_t mst_tc_gemm(const mst_tc_gemm_args& a, const mst_tc_choice& choice, cudaStream_t s);
inline mst_status_t mst_tc_gemm(const mst_tc_gemm_args& a, cudaStream_t s) { return mst_tc_gemm(a, mst_tc_choose(a), s); }
bool mst_tc_gemm_usable(const void* A, int64_t lda, const void* B, int64_t ldb);

// cuTensorMapEncodeTiled of the loaded driver (nullptr when it has none) and the SM count of the current device
typedef CUresult (*mst_encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                        const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                        CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
mst_encode_tiled_fn mst_encode_tiled();
int mst_sm_count();

int mst_tc_pick_splits(int64_t tiles, int64_t slots, int64_t kblocks, double out_bytes, int* cut);

// Process-wide scratch buffer for handle-less entry points (grows on demand; growing synchronises the device).
// Calls that use it must not overlap on the GPU.
mst_status_t mst_workspace(size_t bytes, void** ptr);
// The same per purpose (mst_tc_gemm.cu).
enum { MST_WS_SPLIT = 0, MST_WS_COLUMNS = 1, MST_WS_ATTENTION = 2, MST_WS_IMAGE = 3, MST_WS_KINDS = 4 };
mst_status_t mst_workspace_kind(int kind, size_t bytes, void** ptr);
