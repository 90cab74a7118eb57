// Mixed-Growing topology update (Algorithm 1) on the device.
//
// The three selections of the algorithm (prune by smallest |w|, grow by largest |g|, grow at random) are the same
// primitive: take the k smallest keys of a candidate set, ties broken by the smaller flat index.  Each is done by a
// most-significant-digit radix select (11 bits per pass) that leaves a threshold key tau and the number `rem` of
// entries equal to tau still to take; a popcount + exclusive scan over the mask words then ranks the entries equal to
// tau in flat-index order and the first `rem` of them are taken.  Results are bit masks over the flat index space, so
// the mask rewrite is three bitwise operations per word and the CSR rebuild is the popcount/scan/fill of
// mst_structure.cu.  Integer keys, integer atomics only: the outcome is deterministic and bit-exact.
//
// Two forms, same results: one cooperative launch for the layers of a call (mst_update_fused.cu), and the kernel-per-phase
// sequence below (run_select: one warp per 32-bit mask word, the last block to finish a histogram pass picks the digit; the tie
// ranking is skipped on the device when the threshold key has no surplus ties), which serves layers whose slices do not fit
// the shared memory of the one launch.
#include <cmath>
#include <cstdlib>
#include <new>

#include "mst_bits.cuh"
#include "mst_topology.cuh"

namespace {

enum { MODE_PRUNE = 0, MODE_GRAD = 1, MODE_RAND = 2 };

__device__ __forceinline__ unsigned lanemask_lt() {
  unsigned m;
  asm("mov.u32 %0, %%lanemask_lt;" : "=r"(m));
  return m;
}

template <int MODE>
struct KeyBits {
  static constexpr int value = MODE == MODE_RAND ? 64 : 32;
};
template <int MODE>
struct KeyWord {
  typedef uint32_t type;
};
template <>
struct KeyWord<MODE_RAND> {
  typedef unsigned long long type;
};

// candidate test and key of bit `lane` of word w.  nonfinite is set when a magnitude key is Inf/NaN.
template <int MODE>
__device__ __forceinline__ bool cand_key_w(const SelParams& P, int64_t w, int lane, uint32_t old_word, int32_t old_base,
                                           uint32_t grad_word, unsigned long long& key, bool& nonfinite) {
  // flat index of this bit; when I is a multiple of 32 the mask words tile the flat index space exactly
  long long f;
  bool col_ok = true;
  if (P.aligned) {
    f = (long long)w * 32 + lane;
  } else {
    const unsigned wu = (unsigned)w, wpr = (unsigned)P.wpr;  // nwords < 2^31
    const int o = (int)(wu / wpr), c = (int)(wu - (unsigned)o * wpr) * 32 + lane;
    col_ok = c < P.I;
    f = (long long)o * P.I + c;
  }
  nonfinite = false;
  key = 0;
  if (MODE == MODE_PRUNE) {
    const uint32_t word = old_word;
    if (!((word >> lane) & 1u)) return false;
    const int32_t pos = old_base + __popc(word & lanemask_lt());
    uint32_t k;
    if (P.bf16)
      k = ((uint32_t)(((const uint16_t*)P.vals)[pos] & 0x7FFFu)) << 16;
    else
      k = ((const uint32_t*)P.vals)[pos] & 0x7FFFFFFFu;
    if (P.lambda != 0.f) {  // MEST criterion, fp32 with one rounding per operation (never contracted to an FMA)
      const float g = fabsf(P.G[f]);
      k = __float_as_uint(__fadd_rn(__uint_as_float(k), __fmul_rn(P.lambda, g))) & 0x7FFFFFFFu;
    }
    nonfinite = k >= 0x7F800000u;
    key = k;
    return true;
  } else if (MODE == MODE_GRAD) {
    uint32_t word = ~old_word;
    if (P.allow) word |= P.pruned_bits[w];
    if (!col_ok || !((word >> lane) & 1u)) return false;
    const uint32_t k = __float_as_uint(P.G[f]) & 0x7FFFFFFFu;
    nonfinite = k >= 0x7F800000u;
    key = 0xFFFFFFFFu - k;  // largest magnitude first
    return true;
  } else {
    const uint32_t word = ~old_word & ~grad_word;
    if (!col_ok || !((word >> lane) & 1u)) return false;
    key = sm64_mix(P.stream + SM64_GAMMA * ((unsigned long long)f + 1ULL));
    return true;
  }
}

// same, with the mask words fetched from global memory
template <int MODE>
__device__ __forceinline__ bool cand_key(const SelParams& P, int64_t w, int lane, unsigned long long& key,
                                         bool& nonfinite) {
  const uint32_t ow = P.old_bits[w];
  const int32_t ob = MODE == MODE_PRUNE ? P.old_wscan[w] : 0;
  const uint32_t gw = MODE == MODE_RAND ? P.grad_bits[w] : 0u;
  return cand_key_w<MODE>(P, w, lane, ow, ob, gw, key, nonfinite);
}

constexpr int RADIX_BITS = MST_SELECT_RADIX_BITS;
constexpr int BINS = MST_SELECT_BINS;
constexpr int HIST_THREADS = 1024;
constexpr int BINS_PER_THREAD = BINS / HIST_THREADS;

__host__ __device__ constexpr int num_passes(int key_bits) { return (key_bits + RADIX_BITS - 1) / RADIX_BITS; }
// digit `pass` (most significant first) covers key bits [pass_shift, pass_shift + pass_width)
__host__ __device__ constexpr int pass_shift(int key_bits, int pass) {
  return key_bits - RADIX_BITS * (pass + 1) > 0 ? key_bits - RADIX_BITS * (pass + 1) : 0;
}
__host__ __device__ constexpr int pass_width(int key_bits, int pass) {
  return key_bits - RADIX_BITS * pass < RADIX_BITS ? key_bits - RADIX_BITS * pass : RADIX_BITS;
}

__global__ void select_init(mst_select_state* st, long long k, unsigned int* hist, unsigned int* counter) {
  if (threadIdx.x == 0) {
    st->prefix = 0;
    st->k = k;
    st->tau = 0;
    st->rem = 0;
    st->need_rank = 0;
    st->pad = 0;   // 'done' flag: later passes return at once
    *counter = 0;
  }
  for (int b = threadIdx.x; b < BINS; b += blockDim.x) hist[b] = 0;
}

template <int MODE>
__global__ void __launch_bounds__(HIST_THREADS) select_hist(SelParams P, int pass, mst_select_state* st, unsigned int* hist,
                                                   unsigned int* counter, int32_t* flags) {
  constexpr int KB = KeyBits<MODE>::value;
  __shared__ unsigned int sh[BINS];
  __shared__ unsigned int warp_tot[HIST_THREADS / 32];
  __shared__ bool is_last;
  if (st->pad) return;  // an earlier pass already fixed the threshold
  for (int b = threadIdx.x; b < BINS; b += HIST_THREADS) sh[b] = 0;
  __syncthreads();
  const unsigned long long prefix = st->prefix;
  const int shift = pass_shift(KB, pass);
  const unsigned dmask = (1u << pass_width(KB, pass)) - 1u;
  const int hi_shift = shift + pass_width(KB, pass);  // bits above this digit
  const int lane = threadIdx.x & 31;
  const int64_t warps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  bool saw_nonfinite = false;
  // four words per trip so that their dependent loads (mask word -> position -> value) overlap
  constexpr int BATCH = 4;
  for (int64_t w0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w0 < P.nwords; w0 += warps * BATCH) {
    unsigned digit[BATCH];
    bool live[BATCH];
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
      const int64_t w = w0 + (int64_t)j * warps;
      unsigned long long key = 0;
      bool nf = false;
      const bool c = w < P.nwords && cand_key<MODE>(P, w, lane, key, nf);
      saw_nonfinite |= (c && nf);
      // entries whose higher digits differ from the prefix are out of the race
      live[j] = c && (pass == 0 || (key >> hi_shift) == prefix);
      digit[j] = live[j] ? (unsigned)((key >> shift) & dmask) : (unsigned)BINS;
    }
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
      if (live[j]) atomicAdd(&sh[digit[j]], 1u);
    }
  }
  if (pass == 0 && saw_nonfinite) atomicOr(&flags[0], MST_FLAG_NONFINITE);
  __syncthreads();
  for (int b = threadIdx.x; b < BINS; b += HIST_THREADS)
    if (sh[b]) atomicAdd(&hist[b], sh[b]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = (atomicAdd(counter, 1u) == gridDim.x - 1);
  __syncthreads();
  if (!is_last) return;
  // last block to finish: every other block's contribution is visible; pick the digit that holds the k-th key
  __threadfence();
  unsigned int mine[BINS_PER_THREAD];
  unsigned int tsum = 0;
#pragma unroll
  for (int j = 0; j < BINS_PER_THREAD; ++j) {
    const int b = threadIdx.x * BINS_PER_THREAD + j;
    mine[j] = atomicAdd(&hist[b], 0u);
    hist[b] = 0;  // ready for the next pass
    tsum += mine[j];
  }
  // exclusive prefix of the per-thread sums over the block
  unsigned int incl = tsum;
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) warp_tot[threadIdx.x >> 5] = incl;
  __syncthreads();
  unsigned int before = incl - tsum;
  for (int wv = 0; wv < (int)(threadIdx.x >> 5); ++wv) before += warp_tot[wv];
  const long long k = st->k;
  __syncthreads();  // everyone has read st->k before the owner rewrites it
  const bool owner = (long long)before < k && k <= (long long)before + (long long)tsum;
  if (owner) {
    long long cum = before;
    int bin = 0;
#pragma unroll
    for (int j = 0; j < BINS_PER_THREAD; ++j) {
      if (cum + (long long)mine[j] >= k) { bin = j; break; }
      cum += mine[j];
    }
    const unsigned long long np = (prefix << pass_width(KB, pass)) | (unsigned long long)(threadIdx.x * BINS_PER_THREAD + bin);
    st->prefix = np;
    st->k = k - cum;
    if (shift == 0) {
      st->tau = np;
      st->rem = k - cum;
      st->need_rank = ((long long)mine[bin] > k - cum) ? 1 : 0;  // ties at the threshold beyond what is taken
    } else if ((long long)mine[bin] == k - cum) {
      // every key that shares this prefix is taken: the lower digits cannot matter, stop here
      st->tau = (np << shift) | ((1ULL << shift) - 1ULL);
      st->rem = k - cum;
      st->need_rank = 0;
      st->pad = 1;
    }
  }
  if (threadIdx.x == HIST_THREADS - 1) {
    const long long total = (long long)before + (long long)tsum;
    if (total < k) atomicOr(&flags[0], MST_FLAG_CORRUPT);  // fewer candidates than requested: ruled out by the host counts
    *counter = 0;
  }
}

// cnt[w] = number of candidates in word w whose key equals tau (skipped when no tie has to be ranked)
template <int MODE>
__global__ void __launch_bounds__(256) select_count_equal(SelParams P, const mst_select_state* st,
                                                          int32_t* __restrict__ cnt) {
  if (!st->need_rank) return;
  const unsigned long long tau = st->tau;
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= P.nwords) return;
  unsigned long long key;
  bool nf;
  const bool c = cand_key<MODE>(P, w, lane, key, nf);
  const unsigned eq = __ballot_sync(0xffffffffu, c && key == tau);
  if (lane == 0) cnt[w] = __popc(eq);
}

template <int MODE>
__global__ void __launch_bounds__(256) select_mark(SelParams P, const mst_select_state* st,
                                                   const int32_t* __restrict__ eq_scan, uint32_t* __restrict__ out) {
  const unsigned long long tau = st->tau;
  const long long rem = st->rem;
  const bool need_rank = st->need_rank != 0;
  const int lane = threadIdx.x & 31;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= P.nwords) return;
  unsigned long long key;
  bool nf;
  const bool c = cand_key<MODE>(P, w, lane, key, nf);
  const bool iseq = c && key == tau;
  const unsigned eq = __ballot_sync(0xffffffffu, iseq);
  // without ties beyond the quota every entry equal to tau is taken; otherwise the first `rem` in index order
  const long long rank = need_rank ? (long long)eq_scan[w] + __popc(eq & lanemask_lt()) : -1;
  const bool take = c && (key < tau || (iseq && rank < rem));
  const unsigned bits = __ballot_sync(0xffffffffu, take);
  if (lane == 0) out[w] = bits;
}

__global__ void max_row_nnz(const int32_t* __restrict__ row_ptr, int O, int32_t* flags) {
  const int o = blockIdx.x * blockDim.x + threadIdx.x;
  if (o < O) atomicMax(&flags[1], row_ptr[o + 1] - row_ptr[o]);
}

template <int MODE>
mst_status_t run_select(mst_layer* L, const SelParams& P, int64_t k, uint32_t* out_bits, cudaStream_t s) {
  if (k <= 0) {
    MST_CUDA_TRY(cudaMemsetAsync(out_bits, 0, sizeof(uint32_t) * L->nwords, s));
    return MST_OK;
  }
  constexpr int passes = num_passes(KeyBits<MODE>::value);
  select_init<<<1, 256, 0, s>>>(L->sel, (long long)k, L->hist, L->counter); MST_COUNT_LAUNCH();
  int64_t blocks = (L->nwords * 32 + HIST_THREADS - 1) / HIST_THREADS;
  if (blocks > 2 * 148) blocks = 2 * 148;  // all SMs fully occupied; each block ends with one global add per non-empty bin
  for (int p = 0; p < passes; ++p)
    { select_hist<MODE><<<(unsigned)blocks, HIST_THREADS, 0, s>>>(P, p, L->sel, L->hist, L->counter, L->flags); MST_COUNT_LAUNCH(); }
  const unsigned wgrid = (unsigned)((L->nwords * 32 + 255) / 256);
  select_count_equal<MODE><<<wgrid, 256, 0, s>>>(P, L->sel, L->word_cnt); MST_COUNT_LAUNCH();
  MST_TRY(mst_scan_i32_if(L->word_cnt, L->word_scan, L->nwords, L->block_sums, &L->sel->need_rank, s));
  select_mark<MODE><<<wgrid, 256, 0, s>>>(P, L->sel, L->word_scan, out_bits); MST_COUNT_LAUNCH();
  MST_CUDA_TRY(cudaGetLastError());
  return MST_OK;
}

}  // namespace

extern "C" mst_status_t mst_update_counts(double prune_frac, int64_t nnz, int64_t target_nnz, int64_t numel,
                                          double random_ratio, int64_t counts[4]) {
  if (!counts) return MST_ERR_INVALID_ARG;
  if (!(prune_frac >= 0.0 && prune_frac <= 1.0) || !(random_ratio >= 0.0 && random_ratio <= 1.0))
    return MST_ERR_INVALID_ARG;
  if (nnz < 0 || nnz > numel) return MST_ERR_INVALID_ARG;
  if (target_nnz < 0) target_nnz = nnz;
  if (target_nnz > numel) return MST_ERR_INFEASIBLE;
  // floor(zeta * nnz) in double; then the smallest adjustment that lets the layer reach its target count
  int64_t n_prune = (int64_t)(prune_frac * (double)nnz);
  const int64_t lo = nnz - target_nnz > 0 ? nnz - target_nnz : 0;
  const int64_t hi = nnz < numel - target_nnz ? nnz : numel - target_nnz;
  if (n_prune < lo) n_prune = lo;
  if (n_prune > hi) n_prune = hi;
  const int64_t n_grow = n_prune + target_nnz - nnz;
  const int64_t n_rand = (int64_t)((double)n_grow * random_ratio);
  counts[0] = n_prune;
  counts[1] = n_grow;
  counts[2] = n_rand;
  counts[3] = n_grow - n_rand;
  return MST_OK;
}

extern "C" mst_status_t mst_rand_bracket(int64_t k, int64_t candidates, double sigmas, int64_t list_capacity, uint64_t* lo,
                                         uint64_t* hi, int32_t* planned) {
  if (!lo || !hi || !planned || list_capacity < 0) return MST_ERR_INVALID_ARG;
  *lo = *hi = 0;
  *planned = 0;
  if (k <= 0 || candidates <= 0 || k > candidates || !(sigmas > 0.0)) return MST_OK;   // nothing to bracket, or switched off
  const int64_t m = (int64_t)(sigmas * sqrt((double)k)) + 16;
  if (3 * m > list_capacity) return MST_OK;               // expected list length 2m: leave room for its own spread
  const int64_t lo_cnt = k - m > 0 ? k - m : 0, hi_cnt = k + m;
  const unsigned __int128 one = (unsigned __int128)1 << 64;
  const uint64_t l = (uint64_t)(one * (unsigned __int128)lo_cnt / (unsigned __int128)candidates);
  const uint64_t h = hi_cnt >= candidates ? ~(uint64_t)0 : (uint64_t)(one * (unsigned __int128)hi_cnt / (unsigned __int128)candidates);
  if (h <= l) return MST_OK;
  *lo = l;
  *hi = h;
  *planned = 1;
  return MST_OK;
}

namespace {

// Bracket for the random growth: the n_rand-th smallest of C independent uniform 64-bit keys lies, with probability
// 1 - 1e-8 or better, between the quantiles (k - m) / C and (k + m) / C with m = sigmas * sqrt(k) + 16 (the count of
// keys below a quantile is binomial with a standard deviation below sqrt(k)).  The kernel checks the bracket against
// the exact counts and falls back to the general radix select when it missed, so the choice only affects speed.
void plan_rand_bracket(UpdatePlan& pl) {
  const mst_layer* L = pl.L;
  double sigmas = 6.0;
  if (const char* e = getenv("MST_UPDATE_RAND_SIGMAS")) sigmas = atof(e);
  uint64_t lo = 0, hi = 0;
  int32_t planned = 0;
  pl.rand_lo = pl.rand_hi = 0;
  pl.rand_bracket = 0;
  // candidates: inactive entries the gradient growth left.  The list also takes the candidates below the bracket whose growth
  // by gradient is open during the sweep, less than a tenth of them.
  const int64_t room = L->rand_cap - pl.n_rand / 8;
  if (room <= 0) return;
  if (mst_rand_bracket(pl.n_rand, (L->N - L->nnz) - pl.n_grad, sigmas, room, &lo, &hi, &planned) != MST_OK || !planned) return;
  pl.rand_lo = lo;
  pl.rand_hi = hi;
  pl.rand_bracket = 1;
}

mst_status_t plan_update(mst_layer* L, double prune_frac, const mst_regrow_rule_t* rule, const float* G_dense, UpdatePlan* pl) {
  if (!L || !rule) return MST_ERR_INVALID_ARG;
  if (L->nnz < 0) return MST_ERR_NOT_PACKED;
  int64_t cnt[4];
  MST_TRY(mst_update_counts(prune_frac, L->nnz, rule->target_nnz, L->N, rule->random_ratio, cnt));
  pl->L = L;
  pl->n_prune = cnt[0];
  pl->n_rand = cnt[2];
  pl->n_grad = cnt[3];
  pl->target = rule->target_nnz < 0 ? L->nnz : rule->target_nnz;
  if (pl->target > L->cap) return MST_ERR_CAPACITY;
  if (!(rule->prune_grad_weight >= 0.f)) return MST_ERR_INVALID_ARG;
  if ((pl->n_grad > 0 || (rule->prune_grad_weight != 0.f && pl->n_prune > 0)) && !G_dense) return MST_ERR_INVALID_ARG;
  pl->c = L->cur;
  pl->n = L->cur ^ 1;
  SelParams& P = pl->P;
  P.old_bits = L->bits[pl->c];
  P.old_wscan = L->wscan[pl->c];
  P.vals = L->vals[pl->c];
  P.bf16 = L->dtype == MST_BF16;
  P.G = G_dense;
  P.pruned_bits = L->pruned_bits;
  P.grad_bits = L->grad_bits;
  P.O = L->O;
  P.I = L->I;
  P.wpr = L->wpr;
  P.allow = rule->allow_regrow_pruned ? 1 : 0;
  P.aligned = (L->I % 32 == 0) ? 1 : 0;
  P.lambda = rule->prune_grad_weight;
  P.low_zero = (L->dtype == MST_BF16 && P.lambda == 0.f) ? 16 : 0;
  P.nwords = L->nwords;
  {  // state of the random-growth generator for (seed, step, layer): three chained SplitMix64 first outputs
    const unsigned long long a = sm64_mix(rule->seed + SM64_GAMMA);
    const unsigned long long b = sm64_mix((a ^ rule->step) + SM64_GAMMA);
    P.stream = sm64_mix((b ^ (unsigned long long)(int64_t)L->layer_id) + SM64_GAMMA);
  }
  plan_rand_bracket(*pl);
  return MST_OK;
}

// Host epilogue of an update whose kernels have been enqueued: statistics and error report when asked for, then the
// flip to the new buffer set.  `fused`: the structure was built by the one-launch form.
mst_status_t finish_update(const UpdatePlan& pl, bool fused, mst_update_stats_t* stats, cudaStream_t s) {
  mst_layer* L = pl.L;
  const int n = pl.n;
  const int64_t nnz_before = L->nnz;
  if (stats) {
    { max_row_nnz<<<(L->O + 255) / 256, 256, 0, s>>>(L->row_ptr[n], L->O, L->flags); MST_COUNT_LAUNCH(); }
    int32_t f[4] = {0, 0, 0, 0};
    int32_t total = 0;
    MST_CUDA_TRY(cudaMemcpyAsync(f, L->flags, sizeof(f), cudaMemcpyDeviceToHost, s));
    MST_CUDA_TRY(cudaMemcpyAsync(&total, L->wscan[n] + L->nwords, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
    MST_CUDA_TRY(cudaStreamSynchronize(s));
    stats->nnz_before = nnz_before;
    stats->nnz_after = total;
    stats->n_prune = pl.n_prune;
    stats->n_grad = pl.n_grad;
    stats->n_rand = pl.n_rand;
    stats->max_row_nnz = f[1];
    const bool bad = (f[0] & (MST_FLAG_NONFINITE | MST_FLAG_CORRUPT)) || total != pl.target;
    if (bad) {
      // A rejected update is not applied: the structure built in the other buffer set is dropped and the layer keeps
      // its mask, values and nnz.  The CSC arrays may hold the rejected structure, so the view is rebuilt on next use.
      L->csc_valid = 0;
      L->scratch_clean = 0;
      MST_CUDA_TRY(cudaMemsetAsync(L->flags, 0, sizeof(int32_t), s));  // reported: cleared
      stats->nnz_after = nnz_before;
      return (f[0] & MST_FLAG_NONFINITE) ? MST_ERR_NONFINITE : MST_ERR_CORRUPT;
    }
  }
  L->cur = n;
  L->nnz = pl.target;
  ++L->version;
  if (!fused) MST_TRY(mst_build_csc(L, s));
  return MST_OK;
}

// One kernel per phase: layers whose slices do not fit the shared memory of the one-launch form, and MST_UPDATE_FUSED=0
mst_status_t launch_phases(const UpdatePlan& pl, cudaStream_t s) {
  mst_layer* L = pl.L;
  MST_CUDA_TRY(cudaMemsetAsync(L->flags + 1, 0, sizeof(int32_t) * 3, s));
  L->scratch_clean = 0;
  MST_TRY(run_select<MODE_PRUNE>(L, pl.P, pl.n_prune, L->pruned_bits, s));
  MST_TRY(run_select<MODE_GRAD>(L, pl.P, pl.n_grad, L->grad_bits, s));
  MST_TRY(run_select<MODE_RAND>(L, pl.P, pl.n_rand, L->rand_bits, s));
  MST_TRY(mst_combine_update_bits(L, pl.n, s));
  return mst_rebuild_from_bits(L, pl.n, nullptr, 0, pl.c, s);
}

// Kernels of the updates of n layers (everything except the host epilogues); fused[i] tells which form layer i took, *done how
// many layers have their kernels enqueued.
mst_status_t launch_updates(const UpdatePlan* plans, int n, char* fused, int* done, cudaStream_t s) {
  bool one_launch = true;
  if (const char* e = getenv("MST_UPDATE_FUSED")) one_launch = (e[0] != '0');
  for (int i = 0; i < n; *done = i) {
    int taken = 0;
    if (one_launch) MST_TRY(mst_launch_fused_update(plans + i, n - i, &taken, s));
    for (int j = 0; j < taken; ++j) fused[i + j] = 1;
    i += taken;
    if (taken == 0) {
      fused[i] = 0;
      MST_TRY(launch_phases(plans[i], s));
      ++i;
    }
  }
  return MST_OK;
}

}  // namespace

extern "C" mst_status_t mst_topology_update(mst_layer_t* L, double prune_frac, const mst_regrow_rule_t* rule,
                                            const float* G_dense, mst_update_stats_t* stats, mst_stream_t stream) {
  cudaStream_t s = (cudaStream_t)stream;
  UpdatePlan pl;
  MST_TRY(plan_update(L, prune_frac, rule, G_dense, &pl));
  char fused = 0;
  int done = 0;
  MST_TRY(launch_updates(&pl, 1, &fused, &done, s));
  return finish_update(pl, fused != 0, stats, s);
}

extern "C" mst_status_t mst_topology_update_many(int32_t n_layers, mst_layer_t* const* layers, const double* prune_frac,
                                                 const mst_regrow_rule_t* rules, const float* const* G_dense,
                                                 mst_update_stats_t* stats, mst_stream_t stream) {
  if (n_layers < 0 || (n_layers > 0 && (!layers || !prune_frac || !rules || !G_dense))) return MST_ERR_INVALID_ARG;
  if (n_layers == 0) return MST_OK;
  cudaStream_t s = (cudaStream_t)stream;
  // every layer is validated before anything is launched: an argument error leaves all layers untouched
  UpdatePlan* plans = new (std::nothrow) UpdatePlan[n_layers];
  char* fused = new (std::nothrow) char[n_layers];
  if (!plans || !fused) { delete[] plans; delete[] fused; return MST_ERR_INVALID_ARG; }
  mst_status_t st = MST_OK;
  for (int i = 0; i < n_layers && st == MST_OK; ++i) {
    st = plan_update(layers[i], prune_frac[i], &rules[i], G_dense[i], &plans[i]);
    for (int j = 0; j < i && st == MST_OK; ++j)
      if (layers[j] == layers[i]) st = MST_ERR_INVALID_ARG;   // a layer may appear once
  }
  int done = 0;
  if (st == MST_OK) st = launch_updates(plans, n_layers, fused, &done, s);
  // host epilogues in order; the first failure is reported, later layers are still finished so that no layer is left
  // with kernels enqueued but its buffer sets not flipped
  for (int j = 0; j < done; ++j) {
    const mst_status_t fj = finish_update(plans[j], fused[j] != 0, stats ? &stats[j] : nullptr, s);
    if (st == MST_OK) st = fj;
  }
  delete[] plans;
  delete[] fused;
  return st;
}
