// Operand preparation for the tensor-core products, everything that one product needs in one launch:
//   image   dense image of W.M from the mask words and the CSR values (one bf16 image, or three bf16 pieces of an fp32 layer)
//   rows    fp32 rows -> three bf16 pieces [3][R][pitch] whose sum is the operand; bf16 rows that the TMA unit does not accept
//           (leading dimension or address) -> the same rows at ones it does
// Rows of more than 32 elements are a multiple of 64 apart: a TMA box row of 128 bytes then lies in one line of the L2 cache instead of
// two.  (2051 x 1023 layer, 1999 tokens: rows 2056 elements apart cost the weight gradient 22 us, 2112 apart 15.)
// Memory-bound, and at the sizes of one layer bound by latency: a thread has the loads of its eight columns in flight together
// (3072 x 768 fp32 image: 10 us with a branch per column, 6 without), and a launch of its own costs 2-3 us.
#include "mst_bits.cuh"
#include "mst_internal.cuh"
#include "mst_tc_gemm.cuh"

namespace {

struct RowsPart {
  const void* in;
  int64_t ld;
  uint32_t R, gpr, blocks;   // rows, groups of eight columns per row of the result
  int C;
  uint16_t* out;
  int64_t piece;             // elements between the pieces (fp32)
  int vec_ok;
};

struct ImagePart {
  const uint32_t* bits;
  const int32_t* wscan;
  uint32_t R, gpr, wpr, blocks;
  const void* vals;
  uint16_t* out;
};

__device__ __forceinline__ uint4 pack8(const uint32_t (&v)[8]) {
  return make_uint4(v[0] | (v[1] << 16), v[2] | (v[3] << 16), v[4] | (v[5] << 16), v[6] | (v[7] << 16));
}

// Eight consecutive columns per thread: their stored values are consecutive in CSR order.  Every element of the image is
// written (+0 where nothing is stored), so it needs no clearing.
template <typename V>
__device__ __forceinline__ void image_group(const ImagePart& P, uint32_t g) {
  const uint32_t r = g / P.gpr, c8 = g - r * P.gpr;
  uint32_t m = 0;
  int32_t pos = 0;
  if ((c8 >> 2) < P.wpr) {   // the pitch may reach beyond the last mask word
    const uint32_t w = r * P.wpr + (c8 >> 2), sh = (c8 & 3u) * 8u;
    const uint32_t word = P.bits[w];
    const int32_t first = P.wscan[w];
    m = (word >> sh) & 0xFFu;
    pos = first + __popc(word & ((1u << sh) - 1u));
  }
  V v[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    v[j] = V(0);
    if ((m >> j) & 1u) v[j] = __ldg((const V*)P.vals + pos + __popc(m & ((1u << j) - 1u)));
  }
  uint16_t* out = P.out + (size_t)g * 8;
  if (sizeof(V) == 4) {
    uint32_t p[3][8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      uint32_t q[3];
      mst_split3((float)v[j], q);
#pragma unroll
      for (int k = 0; k < 3; ++k) p[k][j] = q[k];
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(out + (size_t)k * P.R * P.gpr * 8) = pack8(p[k]);
  } else {
    uint32_t p[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) p[j] = (uint32_t)v[j];
    *reinterpret_cast<uint4*>(out) = pack8(p);
  }
}

__device__ __forceinline__ void rows_group(const RowsPart& P, uint32_t g, float) {
  const uint32_t r = g / P.gpr;
  const int c = (int)(g - r * P.gpr) * 8;
  const float* src = (const float*)P.in + (int64_t)r * P.ld + c;
  float x[8];
  if (P.vec_ok && c + 8 <= P.C) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(src)), b = __ldg(reinterpret_cast<const float4*>(src) + 1);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w; x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) x[j] = c + j < P.C ? __ldg(src + j) : 0.f;
  }
  uint32_t p[3][8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    uint32_t q[3];
    mst_split3(x[j], q);
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k][j] = q[k];
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) *reinterpret_cast<uint4*>(P.out + k * P.piece + (size_t)g * 8) = pack8(p[k]);
}

__device__ __forceinline__ void rows_group(const RowsPart& P, uint32_t g, uint16_t) {
  const uint32_t r = g / P.gpr;
  const int c = (int)(g - r * P.gpr) * 8;
  const uint16_t* src = (const uint16_t*)P.in + (int64_t)r * P.ld + c;
  uint4 v;
  if (c + 8 <= P.C) {
    if ((reinterpret_cast<uintptr_t>(src) & 2u) == 0) {   // whole words
      const uint32_t* w = reinterpret_cast<const uint32_t*>(src);
      v = make_uint4(__ldg(w), __ldg(w + 1), __ldg(w + 2), __ldg(w + 3));
    } else {                                              // half a word, three words, half a word
      const uint32_t* w = reinterpret_cast<const uint32_t*>(src + 1);
      const uint32_t a = __ldg(src), w0 = __ldg(w), w1 = __ldg(w + 1), w2 = __ldg(w + 2), b = __ldg(src + 7);
      v = make_uint4(a | (w0 << 16), __funnelshift_r(w0, w1, 16), __funnelshift_r(w1, w2, 16), (w2 >> 16) | (b << 16));
    }
  } else {
    uint32_t e[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) e[j] = c + j < P.C ? (uint32_t)__ldg(src + j) : 0u;
    v = pack8(e);
  }
  *reinterpret_cast<uint4*>(P.out + (size_t)g * 8) = v;
}

template <typename V>
__global__ void __launch_bounds__(256) prepare_kernel(const ImagePart im, const RowsPart a, const RowsPart b) {
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  uint32_t block = blockIdx.x;
  if (block < im.blocks) {
    const uint32_t g = block * 256 + threadIdx.x;
    if (g < im.R * im.gpr) image_group<V>(im, g);
    return;
  }
  block -= im.blocks;
  const bool second = block >= a.blocks;
  const RowsPart& P = second ? b : a;
  const uint32_t g = (second ? block - a.blocks : block) * 256 + threadIdx.x;
  if (g < P.R * P.gpr) rows_group(P, g, V(0));
}

}  // namespace

mst_status_t mst_prepare(mst_dtype_t dtype, const mst_image_job* image, const mst_rows_job* rows, int n_rows, cudaStream_t s) {
  ImagePart im = {};
  if (image && image->out) {
    const int pitch = mst_row_pitch(image->layer->I);
    im.bits = image->layer->bits[image->layer->cur];
    im.wscan = image->layer->wscan[image->layer->cur];
    im.vals = image->layer->vals[image->layer->cur];
    im.R = (uint32_t)image->layer->O;
    im.gpr = (uint32_t)pitch / 8;
    im.wpr = (uint32_t)image->layer->wpr;
    im.blocks = (im.R * im.gpr + 255) / 256;   // the mask has fewer than 2^31 entries
    im.out = image->out;
  }
  RowsPart part[2] = {};
  int filled = 0;
  // thread indices are 32 bits wide: rows beyond 2^30 groups go into further launches
  for (int k = 0; k < n_rows; ++k) {
    const mst_rows_job& J = rows[k];
    const int64_t pitch = mst_row_pitch(J.C), gpr = pitch / 8, chunk = ((int64_t)1 << 30) / gpr;
    const size_t es = dtype == MST_F32 ? 4 : 2;
    for (int64_t r0 = 0; r0 < J.R; r0 += chunk) {
      if (filled == 2) {
        const unsigned blocks = im.blocks + part[0].blocks + part[1].blocks;
        MST_CUDA_TRY(dtype == MST_F32 ? mst_launch_overlapped(prepare_kernel<float>, dim3(blocks), dim3(256), 0, s, im, part[0], part[1])
                                      : mst_launch_overlapped(prepare_kernel<uint16_t>, dim3(blocks), dim3(256), 0, s, im, part[0], part[1]));
        im.blocks = 0;
        part[0] = part[1] = RowsPart{};
        filled = 0;
      }
      RowsPart& P = part[filled++];
      P.in = (const char*)J.in + (size_t)r0 * J.ld * es;
      P.ld = J.ld;
      P.R = (uint32_t)(J.R - r0 < chunk ? J.R - r0 : chunk);
      P.gpr = (uint32_t)gpr;
      P.blocks = (P.R * P.gpr + 255) / 256;
      P.C = J.C;
      P.out = (uint16_t*)J.out + r0 * pitch;
      P.piece = J.R * pitch;
      P.vec_ok = J.ld % 4 == 0 && (reinterpret_cast<uintptr_t>(J.in) & 15u) == 0;
    }
  }
  const unsigned blocks = im.blocks + part[0].blocks + part[1].blocks;
  if (blocks == 0) return MST_OK;
  MST_CUDA_TRY(dtype == MST_F32 ? mst_launch_overlapped(prepare_kernel<float>, dim3(blocks), dim3(256), 0, s, im, part[0], part[1])
                                : mst_launch_overlapped(prepare_kernel<uint16_t>, dim3(blocks), dim3(256), 0, s, im, part[0], part[1]));
  // only now: a call that fails before its launch (no memory for its rows, say) must not leave an unbuilt image behind as valid
  if (image && image->out && image->out == image->layer->dense_w) {
    image->layer->dense_version = image->layer->version;
    image->layer->dense_epoch = image->layer->values_epoch;
  }
  return MST_OK;
}

// Where the dense image of W.M is, *ld elements between its rows, and the job that builds it (nothing to do: job->out = NULL).
// Without value tracking the image is rebuilt at every call anyway, so it lives in a per-device scratch buffer shared by all
// layers (no per-layer memory; like the other scratch kinds, calls that use it must not overlap on the GPU).  With value
// tracking the layer keeps its own image and reuses it until the mask or the values change.
mst_status_t mst_image(const mst_layer* L, mst_image_job* job, const uint16_t** image, int64_t* ld) {
  job->layer = L;
  job->out = nullptr;
  *ld = mst_row_pitch(L->I);
  if (L->nnz == L->N && L->dtype == MST_BF16 && L->I % 8 == 0) {  // every entry kept: the CSR values are the dense matrix
    *image = (const uint16_t*)L->vals[L->cur];
    *ld = L->I;
    return MST_OK;
  }
  if (L->track_values) {
    MST_TRY(mst_alloc_dense(const_cast<mst_layer*>(L)));
    *image = L->dense_w;
    if (L->dense_version == L->version && L->dense_epoch == L->values_epoch) return MST_OK;
    job->out = L->dense_w;
  } else {
    void* ws = nullptr;
    MST_TRY(mst_workspace_kind(MST_WS_IMAGE, mst_image_bytes(L), &ws));
    job->out = (uint16_t*)ws;
    *image = job->out;
  }
  return MST_OK;
}
