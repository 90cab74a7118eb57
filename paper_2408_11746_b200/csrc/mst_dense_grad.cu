// Contractions over the tokens, dY^T X: the dense gradient for gradient-based growth, G[o, i] = sum_t dY[t, o] * X[t, i]
// (fp32 out), and the operand handling it shares with the weight gradient sampled on the mask.
//
// Both operands are MN-major for the tensor cores as they are stored (dY is [T x O], X is [T x I], the contraction runs over
// T): no transposes.  bf16 operands whose rows start on 16-byte boundaries are read in place, others from an aligned copy;
// fp32 operands are cut into three bf16 pieces (mst_tc_split.cu).
#include "mst_internal.cuh"
#include "mst_tc_gemm.cuh"

mst_status_t mst_tc_gradient(mst_tc_gemm_args a, mst_dtype_t dtype, const void* dY, int64_t lddy, const void* X, int64_t ldx,
                             cudaStream_t s) {
  const int O = (int)a.M, I = (int)a.N;
  const int64_t T = a.K;
  const int ldO = mst_row_pitch(O), ldI = mst_row_pitch(I);
  a.A = dY; a.lda = lddy; a.a_mn_major = 1;
  a.B = X; a.ldb = ldx; a.b_mn_major = 1;
  if (dtype == MST_F32) {
    void* ws = nullptr;
    MST_TRY(mst_workspace_kind(MST_WS_COLUMNS, 6 * (size_t)T * (ldO + ldI), &ws));
    uint16_t* x = (uint16_t*)ws + 3 * (size_t)T * ldO;
    const mst_rows_job jobs[2] = {{dY, lddy, T, O, ws}, {X, ldx, T, I, x}};
    MST_TRY(mst_prepare(dtype, nullptr, jobs, 2, s));
    a.A = ws; a.lda = ldO;
    a.B = x; a.ldb = ldI;
    a.redo.kind = MST_REDO_GRADIENT;
    a.redo.A = dY; a.redo.lda = lddy;
    a.redo.B = X; a.redo.ldb = ldx;
    a.redo.K = T;
    return mst_tc_split(a, s);
  }
  const bool okY = mst_tc_gemm_usable(dY, lddy, dY, lddy), okX = mst_tc_gemm_usable(X, ldx, X, ldx);
  if (!okY || !okX) {
    void* ws = nullptr;
    MST_TRY(mst_workspace_kind(MST_WS_COLUMNS, 2 * (size_t)T * ((okY ? 0 : ldO) + (okX ? 0 : ldI)), &ws));
    uint16_t* at = (uint16_t*)ws;
    mst_rows_job jobs[2];
    int n = 0;
    if (!okY) {
      jobs[n++] = {dY, lddy, T, O, at};
      a.A = at; a.lda = ldO;
      at += (size_t)T * ldO;
    }
    if (!okX) {
      jobs[n++] = {X, ldx, T, I, at};
      a.B = at; a.ldb = ldI;
    }
    MST_TRY(mst_prepare(dtype, nullptr, jobs, n, s));
  }
  a.splits = 0;
  return mst_tc_gemm(a, s);
}

namespace {

// with a layer: its entries of G go to dW as well, *sampled when the contraction has seen to that
mst_status_t dense_grad(const mst_layer* L, const void* dY, int64_t lddy, const void* X, int64_t ldx, int64_t T, int32_t out_features,
                        int32_t in_features, mst_dtype_t dtype, float* G, float* dW, bool* sampled, cudaStream_t s) {
  if (!G || T < 0 || out_features <= 0 || in_features <= 0 || (T > 0 && (!dY || !X))) return MST_ERR_INVALID_ARG;
  if (dtype != MST_F32 && dtype != MST_BF16) return MST_ERR_DTYPE;
  if (lddy < out_features || ldx < in_features) return MST_ERR_SHAPE;
  if (T == 0) {
    MST_CUDA_TRY(cudaMemsetAsync(G, 0, sizeof(float) * (size_t)out_features * in_features, s));
    return MST_OK;
  }
  mst_tc_gemm_args a = {};
  a.M = out_features; a.N = in_features; a.K = T;
  a.epilogue = MST_TC_OUT_F32;
  a.out = G; a.ldc = in_features;
  if (L) {
    a.bits = L->bits[L->cur];
    a.wscan = L->wscan[L->cur];
    a.wpr = L->wpr;
    a.also_sampled = dW;
    a.sampled = sampled;
  }
  return mst_tc_gradient(a, dtype, dY, lddy, X, ldx, s);
}

}  // namespace

extern "C" mst_status_t mst_dense_grad(const void* dY, int64_t lddy, const void* X, int64_t ldx, int64_t T,
                                       int32_t out_features, int32_t in_features, mst_dtype_t dtype, float* G,
                                       mst_stream_t stream) {
  return dense_grad(nullptr, dY, lddy, X, ldx, T, out_features, in_features, dtype, G, nullptr, nullptr, (cudaStream_t)stream);
}

extern "C" mst_status_t mst_dense_grad_dw(const mst_layer_t* L, const void* dY, int64_t lddy, const void* X, int64_t ldx,
                                          int64_t T, float* G_dense, float* dW_vals, mst_stream_t stream) {
  if (!L || !G_dense || !dW_vals) return MST_ERR_INVALID_ARG;
  if (L->nnz < 0) return MST_ERR_NOT_PACKED;
  bool sampled = false;
  MST_TRY(dense_grad(L, dY, lddy, X, ldx, T, L->O, L->I, L->dtype, G_dense, dW_vals, &sampled, (cudaStream_t)stream));
  return sampled ? MST_OK : mst_sddmm_from_dense(L, G_dense, dW_vals, stream);
}
