// The Mixed-Growing topology update of one or several layers in ONE cooperative launch: every layer gets a share of the
// blocks in proportion to its size, its blocks own contiguous slices of its mask words, and four barriers among the blocks of a
// layer separate the phases.
//
//   0  samples    4096 keys of the prune candidates (|w| of the active entries) and of the growth candidates (|g| of the
//                 inactive ones) at jittered, evenly spaced positions
//   -- barrier 0; every block finds, from the sample's order statistics, a bracket [lo, hi) of keys that holds the exact
//                 threshold (four standard deviations of the sample rank on either side)
//                 while barrier 0 fills up: the hash keys of the slice's inactive entries
//   1  sweep      one pass over the gradients and values of the slice: an entry below its bracket is taken, one inside goes to a
//                 list in shared memory (3 to 10 % of the candidates), the rest is never looked at again; the listed keys are
//                 counted in 2048 bins over the bracket
//   -- barrier 1; every block finds the bin of the threshold; the entries of that bin (some tens) go to a global list
//   -- barrier 2; every block finds the entry of the wanted rank by (key, position) in that list: the threshold, ties resolved by
//                 the smaller index.  The random growth's threshold is found the same way among the hash keys inside its planned
//                 bracket; entries whose growth by gradient was still open in phase 1 carry their gradient key along
//   2  marking    new mask words and their population
//   -- barrier 3; scan of the blocks' populations
//   3  fill       column indices and values of the new CSR structure
//
// Selections that this cannot resolve (candidate sets that depend on the prune result, the MEST prune key, a bracket that
// missed, a list that would not fit) take a radix select over the slice, 11 bits of (key, position) per pass: exact
// for any distribution, a sweep and a barrier per pass.  Which form ran never changes the result.
//
// What bounds it: instruction issue in the two sweeps (an inactive entry costs one SplitMix64 hash, two 64-bit products and about
// twenty shifts and logic operations, and 4 bytes of gradient) and, around them, a chain of about fifteen block-wide steps and
// L2 round trips of 1-2 us each that several layers in one launch share.  Four layers of a GPT-2-medium block (12.6 M entries,
// d = 0.1, zeta = 0.3, R = 0.25): 74 us, of which the hashes 14, the gradient and value sweep 20; one of its layers alone
// (4.2 M): 50 us, a layer of 0.6 M 36.  (256 bins over the bracket and a third pass over the bin of some hundred entries: 2 us more.)  The form before, one launch per layer with every key in shared memory and five sweeps between six
// grid-wide barriers, took 238 us for the block.
#include <cmath>
#include <cstdlib>

#include "mst_tc_gemm.cuh"
#include "mst_bits.cuh"
#include "mst_topology.cuh"

namespace {

#ifdef MST_UPD_PROFILE
// phase stamps of block 0 of the last launch (SM clock), read back through mst_update_profile
__device__ long long g_upd_stamps[64];
__device__ int g_upd_nstamps;
#define UPD_STAMP(id)                                    \
  do {                                                   \
    if (blockIdx.x == 0 && threadIdx.x == 0) {           \
      const int at_ = g_upd_nstamps;                     \
      if (at_ < 31) {                                    \
        g_upd_stamps[2 * at_] = (id);                    \
        g_upd_stamps[2 * at_ + 1] = clock64();           \
        g_upd_nstamps = at_ + 1;                         \
      }                                                  \
    }                                                    \
  } while (0)
#else
#define UPD_STAMP(id) do { } while (0)
#endif

constexpr int UT = 1024, UW = UT / 32;     // threads and warps of a block; one block per SM
constexpr int UBINS = 2048;                // bins of a block's own histograms and of the radix select
constexpr int USAMPLES = 4096;             // per selection
constexpr int UCOARSE = UBINS;             // bins over a bracket that the blocks of a layer sum up: so many that the threshold's holds a few tens of entries
constexpr int UFEW = 256;                  // entries of the threshold's bin that the warps rank directly
constexpr int UBIN_LIST = 4 * UT;          // entries of the threshold's bin, four per thread
constexpr int UNARROW = UBINS / 2;         // of them, entries that are compared one by one
constexpr int URAND_LOCAL = 1024;          // random candidates inside the bracket, per block
constexpr int ULAYERS = 8;                 // layers per launch
constexpr uint32_t UKEY_END = 0x80000000u; // keys have 31 bits
constexpr uint32_t USPIN = 4u * 1000u * 1000u;

enum { C_BARRIER = 0, C_EXIT = 1, C_BELOW = 2 /*, 3*/, C_LIST = 4 /*, 5*/, C_RBELOW = 6, C_RLIST = 7, C_OVERFLOW = 8, C_WORDS = 64 };

struct ULayer {
  const uint32_t* old_bits;
  const int32_t* old_wscan;
  const void* vals;
  const float* G;
  unsigned long long stream, rand_lo, rand_hi;
  uint32_t* new_bits;
  int32_t *new_wscan, *new_row_ptr, *bsums, *flags;
  uint16_t* new_col;
  void* new_vals;
  unsigned int* hist;              // [2][UCOARSE] bins of the two brackets (in the first 2 * UBINS), then [3][UBINS] rotating for the radix select
  unsigned int* ctr;               // [C_WORDS]; all zero at launch and again at exit, like the histograms
  uint32_t* samples;               // [2][USAMPLES]
  unsigned long long* bin_list;    // [2][UBIN_LIST] (key << 32 | position)
  unsigned long long* rand_list;   // [rand_cap][2]: hash key; gradient key << 32 | slot
  long long n_prune, n_grad, n_rand, nnz, candidates;   // candidates: inactive entries
  float lambda;
  uint32_t nwords;
  int O, I, wpr, bf16, allow, rand_bracket, rand_cap;
  int block0, blocks;              // this layer's share of the grid
};
struct UParams {
  int n, words_cap, list_cap;      // mask words of the largest slice, entries of the shared list
  ULayer L[ULAYERS];
};

// per-block state in shared memory besides the slice
struct UShared {
  unsigned int hist[2][UBINS];
  unsigned int warp_tot[2][UW];
  unsigned long long rlocal[URAND_LOCAL][2];
  int n_rlocal;
  unsigned int below[2], rbelow, overflow;
  uint32_t lo[2], hi[2];                        // brackets (0: prune, 1: gradient)
  uint32_t kmin[2], kmax[2];                    // extreme sample keys
  int stat_bin[4];
  uint32_t span[2][4];                          // smallest and largest key, smallest and largest position of a list
  int small_n[2], small_bin[2], small_rank[2];
  uint32_t bin[2];
  long long bin_rank[2];
  int fast[2];                                  // the selection's threshold was found from its bracket
  unsigned long long tau[2];                    // (key, position) of the last entry taken
  unsigned long long rtau;
  int r_ok, r_bin, r_n;
  long long r_rank;
  unsigned int r_below;
  // radix select
  unsigned long long g_prefix;
  long long g_k;
  int g_state;
  unsigned int abort;
};

struct USlice {
  uint32_t* old;    // mask words before the update
  int32_t* base;    // position of a word's first entry in the value array
  uint32_t* grad;   // entries grown by gradient
  uint32_t* prn;    // entries pruned; later the position of a word's first entry in the new structure
  uint32_t* hc;     // inactive entries whose hash lies below the bracket's upper end; later the new mask words
  unsigned long long* list;   // this warp's entries inside the brackets: gradient from the front, prune from the back
};

// exclusive prefix over the block in thread order; two independent sums at once
__device__ __forceinline__ void u_scan2(unsigned int a, unsigned int b, unsigned int& ea, unsigned int& eb, UShared& sh) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned int x = a, y = b;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int tx = __shfl_up_sync(0xffffffffu, x, o), ty = __shfl_up_sync(0xffffffffu, y, o);
    if (lane >= o) { x += tx; y += ty; }
  }
  __syncthreads();   // the totals are free
  if (lane == 31) { sh.warp_tot[0][warp] = x; sh.warp_tot[1][warp] = y; }
  __syncthreads();
  unsigned int wa = sh.warp_tot[0][lane], wb = sh.warp_tot[1][lane];   // UW == 32: one total per lane
  const unsigned int ta = wa, tb = wb;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int tx = __shfl_up_sync(0xffffffffu, wa, o), ty = __shfl_up_sync(0xffffffffu, wb, o);
    if (lane >= o) { wa += tx; wb += ty; }
  }
  ea = x - a + __shfl_sync(0xffffffffu, wa - ta, warp);
  eb = y - b + __shfl_sync(0xffffffffu, wb - tb, warp);
}

// Barrier among the blocks of one layer (all resident: cooperative launch).  Bounded: on expiry the block raises its abort word,
// records an error and leaves the kernel without touching the new structure any further.
__device__ __forceinline__ void u_arrive(const ULayer& L, UShared& sh) {
  __syncthreads();
  if (threadIdx.x == 0 && !sh.abort) {
    __threadfence();
    atomicAdd(&L.ctr[C_BARRIER], 1u);
  }
}
__device__ __forceinline__ bool u_wait(const ULayer& L, int& count, UShared& sh) {
  ++count;
  if (threadIdx.x == 0 && !sh.abort) {
    const unsigned int want = (unsigned)count * (unsigned)L.blocks;
    uint32_t it = 0;
    while (true) {
      unsigned int v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(&L.ctr[C_BARRIER]) : "memory");
      if (v >= want) break;
      if (++it > USPIN) {
        sh.abort = 1;
        atomicOr(&L.flags[0], MST_FLAG_CORRUPT);
        break;
      }
      if (it > 64) __nanosleep(32);
    }
  }
  __syncthreads();
  return sh.abort == 0;
}
__device__ __forceinline__ bool u_barrier(const ULayer& L, int& count, UShared& sh) {
  u_arrive(L, sh);
  return u_wait(L, count, sh);
}

__device__ __forceinline__ uint32_t u_prune_key(const ULayer& L, uint32_t pos) {
  return (L.bf16 ? (uint32_t)((const uint16_t*)L.vals)[pos] << 16 : ((const uint32_t*)L.vals)[pos]) & 0x7FFFFFFFu;
}
// gradient keys: largest magnitude first
__device__ __forceinline__ uint32_t u_grad_key(float g) { return 0x7FFFFFFFu - (__float_as_uint(g) & 0x7FFFFFFFu); }
constexpr uint32_t U_FIRST_FINITE_GRAD = 0x7FFFFFFFu - 0x7F800000u + 1u;

__device__ __forceinline__ long long u_flat(const ULayer& L, uint32_t w, int lane) {
  const uint32_t o = w / (uint32_t)L.wpr;
  return (long long)w * 32 + lane - (long long)o * (L.wpr * 32 - L.I);
}
__device__ __forceinline__ unsigned long long u_hash(const ULayer& L, uint32_t w, int lane) {
  return sm64_mix(L.stream + SM64_GAMMA * ((unsigned long long)u_flat(L, w, lane) + 1ULL));
}

// ---- phase 0: samples and brackets ----------------------------------------------------------------------------------------
__device__ __forceinline__ void u_write_samples(const ULayer& L, int blk, bool wantA, bool wantB) {
  for (int i = blk + L.blocks * (int)threadIdx.x; i < USAMPLES; i += L.blocks * UT) {
    const uint32_t jitter = (uint32_t)(sm64_mix(L.stream + (unsigned long long)i) >> 48);   // 16 bits
    const unsigned long long at = ((unsigned long long)i << 16) | jitter;                   // 28 bits, evenly spaced
    if (wantA) L.samples[i] = u_prune_key(L, (uint32_t)((at * (unsigned long long)L.nnz) >> 28));
    if (wantB) {
      const uint32_t slot = (uint32_t)((at * ((unsigned long long)L.nwords * 32ULL)) >> 28);
      const uint32_t w = slot >> 5, bit = slot & 31u;
      const bool inside = (w % (uint32_t)L.wpr) * 32u + bit < (uint32_t)L.I;
      uint32_t key = 0xFFFFFFFFu;   // no candidate
      if (inside && !((L.old_bits[w] >> bit) & 1u)) key = u_grad_key(L.G[u_flat(L, w, (int)bit)]);
      L.samples[USAMPLES + i] = key;
    }
  }
}

// Brackets of both selections from the samples (every block, same result) into sh.lo / sh.hi, four standard deviations of the sample
// rank on either side (a threshold outside, once in 10000 updates, costs the radix select; six list half as many entries again): order statistics from 8192 bins on
// the leading 13 key bits (a step of 1/32 octave), prune counts in the low and gradient counts in the high half of a word; the
// lower edge is rounded down, the upper edge up.  `bins`: 8192 words of shared memory, all zero.
constexpr int USTAT_BINS = 8192, USTAT_SHIFT = 18;
__device__ void u_brackets(const ULayer& L, bool wantA, bool wantB, uint32_t* bins, UShared& sh) {
  constexpr int PER = USAMPLES / UT;
  uint32_t ka[PER], kb[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    ka[j] = wantA ? __ldcg(L.samples + j * UT + threadIdx.x) : 0xFFFFFFFFu;
    kb[j] = wantB ? __ldcg(L.samples + USAMPLES + j * UT + threadIdx.x) : 0xFFFFFFFFu;
  }
  uint32_t mn[2] = {0xFFFFFFFFu, 0xFFFFFFFFu}, mx[2] = {0u, 0u};
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    if (ka[j] != 0xFFFFFFFFu) { atomicAdd(&bins[ka[j] >> USTAT_SHIFT], 1u); mn[0] = min(mn[0], ka[j]); mx[0] = max(mx[0], ka[j]); }
    if (kb[j] != 0xFFFFFFFFu) { atomicAdd(&bins[kb[j] >> USTAT_SHIFT], 0x10000u); mn[1] = min(mn[1], kb[j]); mx[1] = max(mx[1], kb[j]); }
  }
#pragma unroll
  for (int s = 0; s < 2; ++s) { mn[s] = __reduce_min_sync(0xffffffffu, mn[s]); mx[s] = __reduce_max_sync(0xffffffffu, mx[s]); }
  if ((threadIdx.x & 31) == 0) {
#pragma unroll
    for (int s = 0; s < 2; ++s) { atomicMin(&sh.kmin[s], mn[s]); atomicMax(&sh.kmax[s], mx[s]); }
  }
  if (threadIdx.x < 4) sh.stat_bin[threadIdx.x] = -1;
  const float qA = L.nnz > 0 ? (float)L.n_prune / (float)L.nnz : 0.f, qB = L.candidates > 0 ? (float)L.n_grad / (float)L.candidates : 0.f;
  __syncthreads();
  constexpr int BPT = USTAT_BINS / UT;   // neighbouring bins per thread
  unsigned int h[BPT], sum = 0;
  const int b0 = BPT * (int)threadIdx.x;
#pragma unroll
  for (int j = 0; j < BPT; j += 4) {
    const uint4 v = *reinterpret_cast<const uint4*>(bins + b0 + j);
    h[j] = v.x; h[j + 1] = v.y; h[j + 2] = v.z; h[j + 3] = v.w;
  }
#pragma unroll
  for (int j = 0; j < BPT; ++j) sum += h[j];   // halves stay below 65536: at most USAMPLES each
  unsigned int e, dummy;
  u_scan2(sum, 0u, e, dummy, sh);
  if (threadIdx.x == UT - 1) sh.r_n = (int)((e + sum) >> 16);
  __syncthreads();
  // 1-based ranks: prune lo, prune hi, gradient lo, gradient hi (0 or beyond the count: open end)
  const int n_valid[2] = {wantA ? USAMPLES : 0, sh.r_n};
  int rank[4];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const float n = (float)n_valid[s], q = s ? qB : qA;
    const int at = (int)(n * q), m = (int)(4.0f * sqrtf(fmaxf(n * q * (1.0f - q), 0.f))) + 4;
    rank[2 * s] = at - m;
    rank[2 * s + 1] = at + m + 1;
  }
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int sft = (s >> 1) * 16;
    int at = (int)((e >> sft) & 0xFFFFu);
    if (rank[s] > at && rank[s] <= at + (int)((sum >> sft) & 0xFFFFu)) {
#pragma unroll
      for (int j = 0; j < BPT; ++j) {
        const int c = (int)((h[j] >> sft) & 0xFFFFu);
        if (rank[s] > at && rank[s] <= at + c) sh.stat_bin[s] = b0 + j;
        at += c;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 2) {
    const int s = threadIdx.x;
    uint32_t lo = 0u, hi = UKEY_END;
    if (rank[2 * s] >= 1 && sh.stat_bin[2 * s] >= 0) lo = (uint32_t)sh.stat_bin[2 * s] << USTAT_SHIFT;
    if (rank[2 * s + 1] <= n_valid[s] && sh.stat_bin[2 * s + 1] >= 0) hi = (uint32_t)(sh.stat_bin[2 * s + 1] + 1) << USTAT_SHIFT;
    if (s == 1 && hi < U_FIRST_FINITE_GRAD) hi = U_FIRST_FINITE_GRAD;   // non-finite gradients are met inside or below the bracket
    sh.lo[s] = lo;
    sh.hi[s] = hi;
  }
  __syncthreads();
}

// Bins over a bracket: linear between lo and hi, one bin each for what lies outside (an open end of the bracket is binned between
// the extreme samples only: the key range beyond them is huge and nearly empty).  A range of few distinct keys (bf16 weights
// have 16 zero bits below their key; just-grown weights are all zero) is divided further by position, so that runs of equal keys
// spread over bins.
struct UBinMap {
  uint32_t lo, hi;
  uint32_t kscale;     // inner bin = (key - lo) * kscale / 2^32, or, where there are fewer distinct keys than bins (0),
  int shift, sub;      // ((key - lo) >> shift) * sub + position * sub / positions
  uint32_t scale;
  __device__ __forceinline__ uint32_t bin(uint32_t key, uint32_t pos) const {
    if (key < lo) return 0u;
    if (key >= hi) return UCOARSE - 1;
    return 1u + (kscale ? __umulhi(key - lo, kscale) : ((key - lo) >> shift) * (uint32_t)sub + __umulhi(pos, scale));
  }
};
__device__ __forceinline__ UBinMap u_bin_map(uint32_t lo, uint32_t hi, uint32_t kmin, uint32_t kmax, int low_zero,
                                             unsigned long long positions) {
  UBinMap m;
  if (lo == 0u && kmin != 0xFFFFFFFFu && kmin < hi) lo = kmin;
  if (hi == UKEY_END && kmax >= lo && kmax < UKEY_END) hi = kmax + 1u;
  m.lo = (lo >> low_zero) << low_zero;
  m.hi = hi;
  const uint32_t span = hi > m.lo ? hi - 1u - m.lo : 0u;
  m.shift = low_zero;
  m.kscale = 0u;
  uint32_t sub = 1;
  if (span >> low_zero >= UCOARSE - 2) {
    m.kscale = (uint32_t)(((unsigned long long)(UCOARSE - 2) << 32) / ((unsigned long long)span + 1ULL));
  } else {
    sub = (UCOARSE - 2) / ((span >> low_zero) + 1u);
    if (positions < 2) sub = 1;
    else if ((unsigned long long)sub >= positions) sub = (uint32_t)(positions - 1);
    if (sub < 1u) sub = 1;
  }
  m.sub = (int)sub;
  m.scale = positions < 2 ? 0u : (uint32_t)(((unsigned long long)m.sub << 32) / positions);
  return m;
}

// ---- phase 1: the sweep ------------------------------------------------------------------------------------------------------
// Entries inside the brackets go to the warp's own part of the list, so that appending is a ballot and a predicated store; n[0] and
// n[1] count the prune entries (from the back) and the gradient entries (from the front).  A part that overflows is noticed by
// the counts.
__device__ __forceinline__ void u_append(bool in, unsigned m, int sel, int& n, int cap, uint32_t key, uint32_t at, const USlice& S) {
  const int i = n + __popc(m & mst_lanemask_lt());
  if (in && i < cap) S.list[sel ? i : cap - 1 - i] = ((unsigned long long)key << 32) | at;
  n += __popc(m);
}

// Random candidates of the slice: the inactive entries whose hash can be below the bracket's upper end (S.hc).  Needs nothing from
// the other blocks and runs while barrier 0 fills up.  Four neighbouring columns per lane.
__device__ void u_hash_sweep(const ULayer& L, uint32_t lo_w, int nloc, const USlice& S) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int pad = L.wpr * 32 - L.I;
  // the last xor-shift of the hash changes only the lowest bit of its high word, so this test admits every hash below rand_hi
  const uint32_t r_test = (uint32_t)(L.rand_hi >> 32) | 1u;
  const uint32_t wpr = (uint32_t)L.wpr;
  const int I = L.I, sub = lane >> 3, nib = (lane & 7) * 4;
  const unsigned long long z0 = L.stream + SM64_GAMMA;
#pragma unroll 2
  for (int l0 = warp * 4; l0 < nloc; l0 += UW * 4) {
    const int li = l0 + sub;
    const uint32_t w = lo_w + (uint32_t)li;
    uint32_t cand = li < nloc ? ((~S.old[li]) >> nib) & 15u : 0u;
    unsigned long long f = w * 32u + (uint32_t)nib;
    if (pad) {
      const uint32_t o = w / wpr;
      f -= (unsigned long long)o * (unsigned)pad;
      const int left = I - (int)((w - o * wpr) * 32u) - nib;   // columns of the row from here on
      cand &= left >= 4 ? 15u : left > 0 ? (1u << left) - 1u : 0u;
    }
    const unsigned long long z = z0 + SM64_GAMMA * f;
    uint32_t h4 = 0u;
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if ((uint32_t)(sm64_mix_top(z + SM64_GAMMA * (unsigned long long)j) >> 32) <= r_test) h4 |= 1u << j;
    h4 &= cand;
    if (h4) atomicOr(&S.hc[li], h4 << nib);
  }
}

__device__ void u_sweep(const ULayer& L, uint32_t lo_w, int nloc, bool fastA, bool fastB, bool fastR, int cap, const USlice& S,
                        UShared& sh, int (&n)[2]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  bool nonfinite = false;
  int below = 0, rbelow = 0;
  if (fastB) {
    // A lane takes four neighbouring columns, eight lanes a mask word: one 16-byte load and one test of the four magnitudes
    // against the bracket's outer edge settle most groups.
    const int pad = L.wpr * 32 - L.I;
    const uint32_t gl = sh.lo[1], outer = UKEY_END - sh.hi[1];   // |g| bits at or above it: inside or sure
    const uint32_t wpr = (uint32_t)L.wpr;
    const int I = L.I;
    const float* __restrict__ G = L.G;
    const bool vec = pad == 0 && (reinterpret_cast<uintptr_t>(G) & 15u) == 0;
    const int sub = lane >> 3, nib = (lane & 7) * 4;
    constexpr int U = 4;   // groups of four words per trip
    for (int l0 = warp * 4; l0 < nloc; l0 += UW * 4 * U) {
      uint32_t cand[U], slot[U], gb[U][4];
      unsigned long long f[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int li = l0 + u * UW * 4 + sub;
        const uint32_t w = lo_w + (uint32_t)li;
        cand[u] = li < nloc ? ((~S.old[li]) >> nib) & 15u : 0u;
        slot[u] = w * 32u + (uint32_t)nib;
        f[u] = slot[u];
        if (pad) {
          const uint32_t o = w / wpr;
          f[u] -= (unsigned long long)o * (unsigned)pad;
          const int left = I - (int)((w - o * wpr) * 32u) - nib;   // columns of the row from here on
          cand[u] &= left >= 4 ? 15u : left > 0 ? (1u << left) - 1u : 0u;
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) gb[u][j] = 0u;
        if (cand[u]) {
          if (vec) {
            const uint4 v = __ldg(reinterpret_cast<const uint4*>(G + f[u]));
            gb[u][0] = v.x; gb[u][1] = v.y; gb[u][2] = v.z; gb[u][3] = v.w;
          } else {
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if ((cand[u] >> j) & 1u) gb[u][j] = __float_as_uint(__ldg(G + f[u] + j));
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int li = l0 + u * UW * 4 + sub;
#pragma unroll
        for (int j = 0; j < 4; ++j) gb[u][j] &= 0x7FFFFFFFu;
        uint32_t hit4 = 0u, sure4 = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (gb[u][j] >= outer) hit4 |= 1u << j;
        hit4 &= cand[u];
        while (__any_sync(0xffffffffu, hit4 != 0u)) {   // one or two rounds: a lane's entries inside or below the bracket, one at a time
          const int j = __ffs(hit4) - 1;
          const uint32_t key = 0x7FFFFFFFu - (j == 0 ? gb[u][0] : j == 1 ? gb[u][1] : j == 2 ? gb[u][2] : gb[u][3]);
          const bool sure = hit4 && key < gl, in = hit4 && !sure;
          nonfinite |= hit4 && key < U_FIRST_FINITE_GRAD;
          if (sure) sure4 |= 1u << j;
          u_append(in, __ballot_sync(0xffffffffu, in), 1, n[1], cap, key, slot[u] + (uint32_t)j, S);
          hit4 &= hit4 - 1;
        }
        if (sure4) {
          atomicOr(&S.grad[li], sure4 << nib);
          below += __popc(sure4);
        }
      }
    }
  }
  below = (int)__reduce_add_sync(0xffffffffu, (unsigned)below);
  if (lane == 0 && below) atomicAdd(&sh.below[1], (unsigned)below);
  if (fastA) {
    // the values of the slice are one contiguous run in CSR order, and positions are ordered like slots
    const uint32_t p0 = nloc > 0 ? (uint32_t)S.base[0] : 0u, p1 = nloc > 0 ? (uint32_t)S.base[nloc - 1] + (uint32_t)__popc(S.old[nloc - 1]) : 0u;
    const uint32_t pl = sh.lo[0], pw = sh.hi[0] - sh.lo[0];
    int belowA = 0;
    constexpr int U = 4;
    for (uint32_t q = p0 + (uint32_t)warp * 32u; q < p1; q += UT * U) {   // uniform over the warp
      uint32_t key[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const uint32_t pos = q + j * UT + lane;
        key[j] = pos < p1 ? u_prune_key(L, pos) : 0xFFFFFFFFu;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        nonfinite |= key[j] >= 0x7F800000u && key[j] != 0xFFFFFFFFu;
        const bool sure = key[j] < pl, in = !sure && key[j] - pl < pw;
        belowA += __popc(__ballot_sync(0xffffffffu, sure));
        u_append(in, __ballot_sync(0xffffffffu, in), 0, n[0], cap, key[j], q + j * UT + lane, S);
      }
    }
    if (lane == 0 && belowA) atomicAdd(&sh.below[0], (unsigned)belowA);
  }
  if (nonfinite) atomicOr(&L.flags[0], MST_FLAG_NONFINITE);
  if (!fastR) return;
  __syncthreads();
  // random candidates that the gradient has not surely taken, one thread per word (one entry in a hundred at the usual counts):
  // below the bracket they are counted, inside it, or with their growth by gradient still open, listed
  const uint32_t gl = sh.lo[1], gw = fastB ? sh.hi[1] - sh.lo[1] : 0u;
  for (int li = threadIdx.x; li < nloc; li += UT) {
    const uint32_t w = lo_w + (uint32_t)li;
    uint32_t m = S.hc[li] & ~S.grad[li], keep = 0;
    while (m) {
      const int b = __ffs(m) - 1;
      m &= m - 1;
      const long long f = u_flat(L, w, b);
      const uint32_t key = fastB ? u_grad_key(__ldg(L.G + f)) : 0xFFFFFFFFu;
      const unsigned long long h = sm64_mix(L.stream + SM64_GAMMA * ((unsigned long long)f + 1ULL));
      if (h >= L.rand_hi) continue;
      keep |= 1u << b;
      const bool open = key - gl < gw;
      if (h >= L.rand_lo || open) {
        const int at = atomicAdd(&sh.n_rlocal, 1);
        if (at < URAND_LOCAL) {
          sh.rlocal[at][0] = h;
          sh.rlocal[at][1] = ((unsigned long long)(open ? key : 0xFFFFFFFFu) << 32) | (w * 32u + (uint32_t)b);
        }
      } else {
        ++rbelow;
      }
    }
    S.hc[li] = keep;
  }
  rbelow = (int)__reduce_add_sync(0xffffffffu, (unsigned)rbelow);
  if (lane == 0 && rbelow) atomicAdd(&sh.rbelow, (unsigned)rbelow);
}

// ---- radix select over the slice: exact threshold of any selection ----------------------------------------------------------------
// The k-th smallest of the candidates' 64-bit keys, 11 bits per pass: (key << 32 | slot) for the magnitudes, which makes ties
// a matter of the smaller index, the hash for the random growth.  All keys differ, so the pass that leaves one bin with exactly
// the entries still wanted ends it.
enum { U_PRUNE = 0, U_GRAD = 1, U_RAND = 2 };
template <int MODE>
__device__ bool u_radix_select(const ULayer& L, int blk, uint32_t lo_w, int nloc, long long k, int& barriers, int& gpass, const USlice& S,
                               UShared& sh, unsigned long long& tau) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b0 = 2 * (int)threadIdx.x;
  __syncthreads();
  if (threadIdx.x == 0) { sh.g_prefix = 0; sh.g_k = k; sh.g_state = 0; }
  bool nonfinite = false;
  for (int pass = 0, top = 64; top > 0; ++pass) {
    const int width = top >= 11 ? 11 : top, shift = top - width;
    for (int b = threadIdx.x; b < UBINS; b += UT) sh.hist[0][b] = 0u;
    __syncthreads();
    const unsigned long long prefix = sh.g_prefix;
    for (int li = warp; li < nloc; li += UW) {
      const uint32_t w = lo_w + (uint32_t)li, old = S.old[li];
      const bool inside = (int)((w % (uint32_t)L.wpr) * 32u) + lane < L.I;
      bool cand;
      unsigned long long key = 0;
      if (MODE == U_PRUNE) {
        cand = (old >> lane) & 1u;
        if (cand) {
          uint32_t kk = u_prune_key(L, (uint32_t)S.base[li] + (uint32_t)__popc(old & ((1u << lane) - 1u)));
          if (L.lambda != 0.f) {  // MEST criterion, fp32 with one rounding per operation (never contracted to an FMA)
            const float g = fabsf(L.G[u_flat(L, w, lane)]);
            kk = __float_as_uint(__fadd_rn(__uint_as_float(kk), __fmul_rn(L.lambda, g))) & 0x7FFFFFFFu;
          }
          if (pass == 0) nonfinite |= kk >= 0x7F800000u;
          key = ((unsigned long long)kk << 32) | (w * 32u + (uint32_t)lane);
        }
      } else if (MODE == U_GRAD) {
        cand = inside && (((~old | (L.allow ? S.prn[li] : 0u)) >> lane) & 1u);
        if (cand) {
          const uint32_t kk = u_grad_key(L.G[u_flat(L, w, lane)]);
          if (pass == 0) nonfinite |= kk < U_FIRST_FINITE_GRAD;
          key = ((unsigned long long)kk << 32) | (w * 32u + (uint32_t)lane);
        }
      } else {
        cand = inside && ((~(old | S.grad[li]) >> lane) & 1u);
        if (cand) key = u_hash(L, w, lane);
      }
      if (cand && (top == 64 || (key >> top) == prefix)) atomicAdd(&sh.hist[0][(unsigned)(key >> shift) & ((1u << width) - 1u)], 1u);
    }
    __syncthreads();
    unsigned int* gh = L.hist + (2 + gpass % 3) * UBINS;
    for (int b = threadIdx.x; b < UBINS; b += UT) {
      const unsigned int v = sh.hist[0][b];
      if (v) atomicAdd(&gh[b], v);
    }
    if (!u_barrier(L, barriers, sh)) return false;
    const unsigned int h0 = __ldcg(gh + b0), h1 = __ldcg(gh + b0 + 1);
    unsigned int e, dummy;
    u_scan2(h0 + h1, 0u, e, dummy, sh);
    const long long kk = sh.g_k;
    __syncthreads();
    const bool first = (long long)e < kk && kk <= (long long)e + h0, second = (long long)e + h0 < kk && kk <= (long long)e + h0 + h1;
    if (first || second) {
      sh.g_prefix = (top == 64 ? 0ULL : prefix << width) | (unsigned long long)(b0 + (second ? 1 : 0));
      const long long left = kk - e - (second ? (long long)h0 : 0);
      sh.g_k = left;
      sh.g_state = ((long long)(second ? h1 : h0) == left) ? 2 : 1;
    }
    if (blk == 0) {   // the buffer two passes ahead was last read before this barrier
      unsigned int* gz = L.hist + (2 + (gpass + 2) % 3) * UBINS;
      for (int b = threadIdx.x; b < UBINS; b += UT) gz[b] = 0u;
    }
    ++gpass;
    __syncthreads();
    const int state = sh.g_state;
    const unsigned long long np = sh.g_prefix;
    __syncthreads();
    if (threadIdx.x == 0) sh.g_state = 0;
    if (state == 0) {   // fewer candidates than wanted (ruled out by the host's counts): take everything
      if (blk == 0 && threadIdx.x == 0) atomicOr(&L.flags[0], MST_FLAG_CORRUPT);
      tau = ~0ULL;
      break;
    }
    tau = shift ? (np << shift) | ((1ULL << shift) - 1ULL) : np;
    if (state == 2) break;
    top = shift;
  }
  if (nonfinite) atomicOr(&L.flags[0], MST_FLAG_NONFINITE);
  return true;
}

// ---- behind barrier 1: the bin of the threshold; its entries go to the layer's list -------------------------------------------
__device__ void u_pick_bins(const ULayer& L, const bool (&want)[2], const UBinMap& mapA, const UBinMap& mapB, const int (&cnt)[2], int cap, const USlice& S,
                            UShared& sh) {
  const int b0 = 2 * (int)threadIdx.x;
  const uint2 a = __ldcg(reinterpret_cast<const uint2*>(L.hist) + threadIdx.x), c = __ldcg(reinterpret_cast<const uint2*>(L.hist + UCOARSE) + threadIdx.x);
  const unsigned int a0 = a.x, a1 = a.y, c0 = c.x, c1 = c.y;
  const unsigned int overflow = __ldcg(L.ctr + C_OVERFLOW), below[2] = {__ldcg(L.ctr + C_BELOW), __ldcg(L.ctr + C_BELOW + 1)};
  unsigned int eA, eB;
  u_scan2(a0 + a1, c0 + c1, eA, eB, sh);
  if (threadIdx.x < 2) { sh.fast[threadIdx.x] = 0; sh.small_n[threadIdx.x] = 0; }
  unsigned long long* stage = reinterpret_cast<unsigned long long*>(sh.hist);   // [2][UNARROW], the bins are not needed any more
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!want[s] || ((overflow >> s) & 1u)) continue;   // uniform over the layer's blocks
    const long long k = (s ? L.n_grad : L.n_prune) - (long long)below[s];   // rank inside the bracket
    const long long e = s ? eB : eA, h0 = s ? c0 : a0, h1 = s ? c1 : a1;
    const bool first = e < k && k <= e + h0, second = e + h0 < k && k <= e + h0 + h1;
    if (first || second) {
      sh.bin[s] = (uint32_t)(b0 + (second ? 1 : 0));
      sh.bin_rank[s] = k - e - (second ? h0 : 0);
      sh.fast[s] = (second ? h1 : h0) <= UBIN_LIST ? 1 : 0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!want[s] || !sh.fast[s]) continue;
    const uint32_t bin = sh.bin[s];
    for (int i = threadIdx.x & 31; i < cnt[s]; i += 32) {
      const unsigned long long v = S.list[s ? i : cap - 1 - i];
      if ((s ? mapB : mapA).bin((uint32_t)(v >> 32), (uint32_t)v) == bin) {
        const int at = atomicAdd(&sh.small_n[s], 1);
        if (at < UNARROW) stage[s * UNARROW + at] = v;
      }
    }
  }
  __syncthreads();
  if (threadIdx.x < 2 && sh.small_n[threadIdx.x] > 0)
    sh.small_bin[threadIdx.x] = (int)atomicAdd(&L.ctr[C_LIST + threadIdx.x], (unsigned)sh.small_n[threadIdx.x]);
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s)
    for (int i = threadIdx.x; i < sh.small_n[s]; i += UT) {
      if (i < UNARROW) L.bin_list[s * UBIN_LIST + sh.small_bin[s] + i] = stage[s * UNARROW + i];
      else atomicOr(&L.ctr[C_OVERFLOW], 1u << s);   // more than a block can stage: the radix select takes over
    }
}

// ---- behind barrier 2: exact thresholds of the selections whose bin was listed ------------------------------------------------
// Few entries, as the bins are made for: half of the warps see to each selection, every one of them holds all of its entries, up to eight a
// lane, and ranks each sixteenth by ballots.  False if there are more.
__device__ __forceinline__ bool u_rank_few(const ULayer& L, UShared& sh) {
  const int lane = threadIdx.x & 31, s = threadIdx.x >> 9, warp = (threadIdx.x >> 5) & 15;
  const unsigned int overflow = __ldcg(L.ctr + C_OVERFLOW), count[2] = {__ldcg(L.ctr + C_LIST), __ldcg(L.ctr + C_LIST + 1)};
  constexpr int PER = UFEW / 32;
  unsigned long long v[PER];   // the places exist whatever the count
#pragma unroll
  for (int h = 0; h < PER; ++h) v[h] = __ldcg(L.bin_list + s * UBIN_LIST + 32 * h + lane);
  if ((overflow & 3u) || (sh.fast[0] && count[0] > UFEW) || (sh.fast[1] && count[1] > UFEW)) return false;   // uniform over the layer's blocks
  const int n = sh.fast[s] ? (int)count[s] : 0, want = (int)sh.bin_rank[s] - 1;
#pragma unroll
  for (int h = 0; h < PER; ++h)
    if (lane + 32 * h >= n) v[h] = ~0ULL;
#pragma unroll
  for (int h = 0; h < PER; ++h) {
#pragma unroll
    for (int half = 0; half < 32; half += 16) {
      if (warp + half + 32 * h >= n) break;
      const unsigned long long x = __shfl_sync(0xffffffffu, v[h], warp + half);
      int rank = 0;
#pragma unroll
      for (int j = 0; j < PER; ++j)
        if (32 * j < n) rank += __popc(__ballot_sync(0xffffffffu, v[j] < x));
      if (rank == want && lane == 0) sh.tau[s] = x;
    }
  }
  __syncthreads();
  return true;
}

// The bin's entries (at most four per thread, in registers) are binned once more between their extremes, by key or, when they all
// have the same key, by position; the entries of the resulting bin are compared with one another.
__device__ void u_rank_bins(const ULayer& L, UShared& sh) {
  constexpr int PER = UBIN_LIST / UT;
  const int lane = threadIdx.x & 31;
  unsigned long long v[2][PER];
  int n[2];
  // the first entry of every thread is fetched together with the counts (its place exists whatever they are)
  const unsigned int overflow = __ldcg(L.ctr + C_OVERFLOW), count[2] = {__ldcg(L.ctr + C_LIST), __ldcg(L.ctr + C_LIST + 1)};
#pragma unroll
  for (int s = 0; s < 2; ++s) v[s][0] = __ldcg(L.bin_list + s * UBIN_LIST + threadIdx.x);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    n[s] = sh.fast[s] && !((overflow >> s) & 1u) ? (int)count[s] : 0;
#pragma unroll
    for (int j = 1; j < PER; ++j) v[s][j] = j * UT + (int)threadIdx.x < n[s] ? __ldcg(L.bin_list + s * UBIN_LIST + j * UT + threadIdx.x) : 0ULL;
  }
  __syncthreads();   // sh.fast has been read
  if (threadIdx.x < 2) {
    if ((overflow >> threadIdx.x) & 1u) sh.fast[threadIdx.x] = 0;
    sh.span[threadIdx.x][0] = sh.span[threadIdx.x][2] = 0xFFFFFFFFu;
    sh.span[threadIdx.x][1] = sh.span[threadIdx.x][3] = 0u;
    sh.small_n[threadIdx.x] = 0;
    sh.small_bin[threadIdx.x] = -1;
  }
  for (int b = threadIdx.x; b < UBINS; b += UT) sh.hist[0][b] = sh.hist[1][b] = 0u;
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if ((int)(threadIdx.x & ~31u) >= n[s]) continue;   // warps without entries
    uint32_t k0 = 0xFFFFFFFFu, k1 = 0u;
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (j * UT + (int)threadIdx.x < n[s]) { k0 = min(k0, (uint32_t)(v[s][j] >> 32)); k1 = max(k1, (uint32_t)(v[s][j] >> 32)); }
    k0 = __reduce_min_sync(0xffffffffu, k0);
    k1 = __reduce_max_sync(0xffffffffu, k1);
    if (lane == 0) { atomicMin(&sh.span[s][0], k0); atomicMax(&sh.span[s][1], k1); }
  }
  __syncthreads();
  const bool tied[2] = {n[0] > 0 && sh.span[0][0] == sh.span[0][1], n[1] > 0 && sh.span[1][0] == sh.span[1][1]};
  if (tied[0] || tied[1]) {   // uniform
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      if (!tied[s] || (int)(threadIdx.x & ~31u) >= n[s]) continue;
      uint32_t p0 = 0xFFFFFFFFu, p1 = 0u;
#pragma unroll
      for (int j = 0; j < PER; ++j)
        if (j * UT + (int)threadIdx.x < n[s]) { p0 = min(p0, (uint32_t)v[s][j]); p1 = max(p1, (uint32_t)v[s][j]); }
      p0 = __reduce_min_sync(0xffffffffu, p0);
      p1 = __reduce_max_sync(0xffffffffu, p1);
      if (lane == 0) { atomicMin(&sh.span[s][2], p0); atomicMax(&sh.span[s][3], p1); }
    }
    __syncthreads();
  }
  uint32_t first[2];
  int shift[2];
  bool by_key[2];
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    by_key[s] = !tied[s];
    first[s] = by_key[s] ? sh.span[s][0] : sh.span[s][2];
    const int bits = 32 - __clz((int)((by_key[s] ? sh.span[s][1] : sh.span[s][3]) - first[s]));
    shift[s] = bits > 11 ? bits - 11 : 0;
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (j * UT + (int)threadIdx.x < n[s]) atomicAdd(&sh.hist[s][((by_key[s] ? (uint32_t)(v[s][j] >> 32) : (uint32_t)v[s][j]) - first[s]) >> shift[s]], 1u);
  }
  __syncthreads();
  {
    const int b0 = 2 * (int)threadIdx.x;
    const unsigned int a0 = sh.hist[0][b0], a1 = sh.hist[0][b0 + 1], c0 = sh.hist[1][b0], c1 = sh.hist[1][b0 + 1];
    unsigned int eA, eB;
    u_scan2(a0 + a1, c0 + c1, eA, eB, sh);
#pragma unroll
    for (int s = 0; s < 2; ++s) {
      const long long k = sh.bin_rank[s], e = s ? eB : eA, h0 = s ? c0 : a0, h1 = s ? c1 : a1;
      const bool one = e < k && k <= e + h0, two = e + h0 < k && k <= e + h0 + h1;
      if (n[s] > 0 && (one || two)) {
        sh.small_bin[s] = b0 + (two ? 1 : 0);
        sh.small_rank[s] = (int)(k - e - (two ? h0 : 0)) - 1;
        if ((two ? h1 : h0) > UNARROW) sh.fast[s] = 0;   // the same in every block: the radix select takes over
      }
    }
  }
  __syncthreads();
  // the histograms' storage now holds the entries that are compared
  unsigned long long* small = reinterpret_cast<unsigned long long*>(sh.hist);
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    if (!sh.fast[s]) continue;   // uniform
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      if (j * UT + (int)threadIdx.x < n[s] &&
          (int)(((by_key[s] ? (uint32_t)(v[s][j] >> 32) : (uint32_t)v[s][j]) - first[s]) >> shift[s]) == sh.small_bin[s])
        small[s * UNARROW + atomicAdd(&sh.small_n[s], 1)] = v[s][j];
    }
  }
  __syncthreads();
#pragma unroll
  for (int s = 0; s < 2; ++s) {
    const int m = sh.fast[s] ? sh.small_n[s] : 0;
    for (int i = threadIdx.x; i < m; i += UT) {
      const unsigned long long x = small[s * UNARROW + i];
      int rank = 0;
      for (int q = 0; q < m; ++q) rank += small[s * UNARROW + q] < x ? 1 : 0;
      if (rank == sh.small_rank[s]) sh.tau[s] = x;
    }
  }
  __syncthreads();
}

// Threshold of the random growth among the listed candidates: those inside the planned bracket, and those below it whose growth by
// gradient was open during the sweep.  False when the bracket missed or a list overflowed (uniform over the layer's blocks).
__device__ bool u_rank_random(const ULayer& L, bool have_grad, UShared& sh) {
  const unsigned int n_list = __ldcg(L.ctr + C_RLIST), overflow = __ldcg(L.ctr + C_OVERFLOW), n_below = __ldcg(L.ctr + C_RBELOW);
  const ulonglong2* list = reinterpret_cast<const ulonglong2*>(L.rand_list);
  const ulonglong2 x0 = __ldcg(list + threadIdx.x);   // the list has room for more entries than a block has threads
  if ((overflow >> 2) & 1u) return false;
  const int n = (int)n_list;
  const unsigned long long gtau = have_grad ? sh.tau[1] : 0ULL, lo = L.rand_lo, range = L.rand_hi - lo;
  const int bshift = (range >> 11) ? 53 - __clzll((long long)range) : 0;   // (key - lo) >> bshift < 2048
  constexpr int PER = 8;   // entries kept in registers by a thread; a longer list is read again
  unsigned long long v[PER];
  __syncthreads();
  for (int b = threadIdx.x; b < UBINS; b += UT) sh.hist[0][b] = 0u;
  if (threadIdx.x == 0) { sh.r_ok = 0; sh.r_n = 0; sh.r_below = 0; }
  __syncthreads();
  unsigned int below = 0, have = 0;
  auto alive = [&](const ulonglong2& x) { return !(have_grad && (x.y >> 32) != 0xFFFFFFFFULL && x.y <= gtau); };   // not grown by gradient
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = j * UT + (int)threadIdx.x;
    v[j] = 0ULL;
    if (i < n) {
      const ulonglong2 x = j == 0 ? x0 : __ldcg(list + i);
      if (alive(x)) {
        if (x.x < lo) ++below;
        else { v[j] = x.x; have |= 1u << j; atomicAdd(&sh.hist[0][(unsigned)((x.x - lo) >> bshift)], 1u); }
      }
    }
  }
  for (int i = PER * UT + (int)threadIdx.x; i < n; i += UT) {
    const ulonglong2 x = __ldcg(list + i);
    if (!alive(x)) continue;
    if (x.x < lo) ++below;
    else atomicAdd(&sh.hist[0][(unsigned)((x.x - lo) >> bshift)], 1u);
  }
  below = __reduce_add_sync(0xffffffffu, below);
  if ((threadIdx.x & 31) == 0 && below) atomicAdd(&sh.r_below, below);
  __syncthreads();
  const long long k = L.n_rand - (long long)n_below - (long long)sh.r_below;   // rank inside the bracket
  const int b0 = 2 * (int)threadIdx.x;
  const unsigned int h0 = sh.hist[0][b0], h1 = sh.hist[0][b0 + 1];
  unsigned int e, dummy;
  u_scan2(h0 + h1, 0u, e, dummy, sh);
  const bool first = (long long)e < k && k <= (long long)e + h0, second = (long long)e + h0 < k && k <= (long long)e + h0 + h1;
  if (first || second) {
    sh.r_bin = b0 + (second ? 1 : 0);
    sh.r_rank = k - e - (second ? (long long)h0 : 0);
    sh.r_ok = (second ? h1 : h0) <= UNARROW ? 1 : 0;   // they must fit the storage of the second histogram
  }
  __syncthreads();
  if (!sh.r_ok) return false;
  const unsigned rbin = (unsigned)sh.r_bin;
  unsigned long long* small = reinterpret_cast<unsigned long long*>(sh.hist[1]);
#pragma unroll
  for (int j = 0; j < PER; ++j)
    if (((have >> j) & 1u) && (unsigned)((v[j] - lo) >> bshift) == rbin) small[atomicAdd(&sh.r_n, 1)] = v[j];
  for (int i = PER * UT + (int)threadIdx.x; i < n; i += UT) {
    const ulonglong2 x = __ldcg(list + i);
    if (alive(x) && x.x >= lo && (unsigned)((x.x - lo) >> bshift) == rbin) small[atomicAdd(&sh.r_n, 1)] = x.x;
  }
  __syncthreads();
  const int m = sh.r_n, r = (int)sh.r_rank - 1;
  for (int i = threadIdx.x; i < m; i += UT) {
    const unsigned long long x = small[i];
    int rank = 0;
    for (int q = 0; q < m; ++q) rank += small[q] < x ? 1 : 0;
    if (rank == r) sh.rtau = x;
  }
  __syncthreads();
  return true;
}

template <typename V>
__device__ void u_fill(const ULayer& L, uint32_t lo_w, int nloc, const USlice& S) {
  const V* old_vals = (const V*)L.vals;
  V* new_vals = (V*)L.new_vals;
  for (int i = threadIdx.x; i < 2 * nloc; i += UT) {   // half a word per thread
    const int li = i >> 1;
    const uint32_t nb = S.hc[li], ob = S.old[li], w = lo_w + (uint32_t)li;
    const uint32_t c0 = (w % (uint32_t)L.wpr) * 32u;
    int32_t pos = (int32_t)S.prn[li] + ((i & 1) ? __popc(nb & 0xFFFFu) : 0);
    const int32_t obase = S.base[li];
    uint32_t m = nb & ((i & 1) ? 0xFFFF0000u : 0xFFFFu);
    while (m) {
      const int b = __ffs(m) - 1;
      m &= m - 1;
      V v = V(0);
      if ((ob >> b) & 1u) v = old_vals[obase + __popc(ob & ((1u << b) - 1u))];
      L.new_col[pos] = (uint16_t)(c0 + b);
      new_vals[pos] = v;
      ++pos;
    }
  }
}

__global__ void __launch_bounds__(UT, 1) mg_update_kernel(const __grid_constant__ UParams P) {
  __shared__ UShared sh;
  extern __shared__ __align__(16) uint32_t s_dyn[];
  mst_grid_launch_dependents();
  mst_grid_dependency_wait();
  int l = 0;
  while (l + 1 < P.n && (int)blockIdx.x >= P.L[l + 1].block0) ++l;
  const ULayer& L = P.L[l];
  const int blk = (int)blockIdx.x - L.block0, lane = threadIdx.x & 31;
  const uint32_t per = (L.nwords + (uint32_t)L.blocks - 1) / (uint32_t)L.blocks;
  const uint32_t lo_w = per * (uint32_t)blk < L.nwords ? per * (uint32_t)blk : L.nwords;
  const int nloc = (int)(lo_w + per < L.nwords ? per : L.nwords - lo_w);
  USlice S;
  const int list_cap = P.list_cap / UW;   // of one warp
  S.list = reinterpret_cast<unsigned long long*>(s_dyn) + (threadIdx.x >> 5) * list_cap;
  S.old = s_dyn + 2 * P.list_cap;
  S.base = reinterpret_cast<int32_t*>(S.old + P.words_cap);
  S.grad = S.old + 2 * P.words_cap;
  S.prn = S.old + 3 * P.words_cap;
  S.hc = S.old + 4 * P.words_cap;

  const bool wantA = L.n_prune > 0, wantB = L.n_grad > 0, wantR = L.n_rand > 0;
  const bool tryA = wantA && L.lambda == 0.f, tryB = wantB && !L.allow;
  const bool tryR = wantR && L.rand_bracket && (tryB || !wantB);   // listed while the gradient growth is settled from its bracket
  for (int i = threadIdx.x; i < nloc; i += UT) {
    S.old[i] = L.old_bits[lo_w + i];
    S.base[i] = L.old_wscan[lo_w + i];
    S.grad[i] = 0u;
    S.hc[i] = 0u;
  }
  if (threadIdx.x < 2) {
    sh.below[threadIdx.x] = 0;
    sh.lo[threadIdx.x] = sh.hi[threadIdx.x] = 0;
    sh.fast[threadIdx.x] = 0;
    sh.tau[threadIdx.x] = 0;
    sh.kmin[threadIdx.x] = 0xFFFFFFFFu;
    sh.kmax[threadIdx.x] = 0u;
  }
  if (threadIdx.x == 0) { sh.n_rlocal = 0; sh.rbelow = 0; sh.overflow = 0; sh.abort = 0; sh.rtau = 0; }
  if (blk == 0 && threadIdx.x < 3) L.flags[1 + threadIdx.x] = 0;   // per-update statistics
#ifdef MST_UPD_PROFILE
  if (blockIdx.x == 0 && threadIdx.x == 0) g_upd_nstamps = 0;
#endif
  UPD_STAMP(1);
  int barriers = 0, gpass = 0;
  bool alive = true, okR = false;

  __syncthreads();   // the slice is in shared memory
  int cnt[2] = {0, 0};   // listed entries of this warp: prune, gradient
  if (tryA || tryB || tryR) {
    if (tryA || tryB) {
      u_write_samples(L, blk, tryA, tryB);
      UPD_STAMP(2);
      u_arrive(L, sh);
    }
    // while the other blocks get there: the slice's gradients on their way to L2, the hashes, the cleared bins of the samples
    if (tryB && nloc > 0) {
      const char* g0 = reinterpret_cast<const char*>(L.G + u_flat(L, lo_w, 0));
      const char* g1 = reinterpret_cast<const char*>(L.G + u_flat(L, lo_w + (uint32_t)nloc - 1, 0));
      for (const char* g = g0 + 128 * (size_t)threadIdx.x; g <= g1; g += 128 * UT) asm volatile("prefetch.global.L2 [%0];" ::"l"(g));
    }
    if (tryR) u_hash_sweep(L, lo_w, nloc, S);
    if (tryA || tryB) {
      for (int i = threadIdx.x; i < USTAT_BINS; i += UT) s_dyn[i] = 0u;
      UPD_STAMP(18);
      alive = u_wait(L, barriers, sh);
      UPD_STAMP(3);
      if (alive) u_brackets(L, tryA, tryB, s_dyn, sh);
      UPD_STAMP(4);
    }
    __syncthreads();
    if (alive) {
      u_sweep(L, lo_w, nloc, tryA, tryB, tryR, list_cap, S, sh, cnt);
      for (int b = threadIdx.x; b < 2 * UCOARSE; b += UT) (&sh.hist[0][0])[b] = 0u;
      __syncthreads();
      UPD_STAMP(5);
    }
    const int low_zero = L.bf16 ? 16 : 0;
    const UBinMap mapA = u_bin_map(sh.lo[0], sh.hi[0], sh.kmin[0], sh.kmax[0], low_zero, (unsigned long long)L.nnz);
    const UBinMap mapB = u_bin_map(sh.lo[1], sh.hi[1], sh.kmin[1], sh.kmax[1], 0, (unsigned long long)L.nwords * 32ULL);
    const bool want[2] = {tryA, tryB};
    const int nr = sh.n_rlocal;
    if (alive) {
      if (threadIdx.x == UT - 1) {   // this block's part of the random list, reserved while the others count
        unsigned int over = nr > URAND_LOCAL ? 4u : 0u;
        if (nr && !over) {
          const unsigned int at = atomicAdd(&L.ctr[C_RLIST], (unsigned)nr);
          if (at + (unsigned)nr > (unsigned)L.rand_cap) over = 4u;
          sh.r_n = (int)at;
        }
        if (sh.below[0]) atomicAdd(&L.ctr[C_BELOW], sh.below[0]);
        if (sh.below[1]) atomicAdd(&L.ctr[C_BELOW + 1], sh.below[1]);
        if (sh.rbelow) atomicAdd(&L.ctr[C_RBELOW], sh.rbelow);
        if (over) {
          atomicOr(&L.ctr[C_OVERFLOW], over);
          atomicOr(&sh.overflow, over);
        }
      }
      if (cnt[0] + cnt[1] <= list_cap) {
        for (int i = lane; i < cnt[1]; i += 32) {
          const unsigned long long v = S.list[i];
          atomicAdd(&sh.hist[1][mapB.bin((uint32_t)(v >> 32), (uint32_t)v)], 1u);
        }
        for (int i = lane; i < cnt[0]; i += 32) {
          const unsigned long long v = S.list[list_cap - 1 - i];
          atomicAdd(&sh.hist[0][mapA.bin((uint32_t)(v >> 32), (uint32_t)v)], 1u);
        }
      } else if (lane == 0) {
        atomicOr(&L.ctr[C_OVERFLOW], 3u);   // both selections then take the radix select
      }
      __syncthreads();
      for (int b = threadIdx.x; b < 2 * UCOARSE; b += UT) {
        const unsigned int v = (&sh.hist[0][0])[b];
        if (v) atomicAdd(&L.hist[b], v);
      }
      if (!(sh.overflow & 4u)) {
        const size_t at = (size_t)sh.r_n;
        for (int i = threadIdx.x; i < 2 * nr; i += UT) L.rand_list[2 * at + i] = (&sh.rlocal[0][0])[i];
      }
      UPD_STAMP(6);
      alive = u_barrier(L, barriers, sh);
      UPD_STAMP(7);
    }
    if (alive) {
      u_pick_bins(L, want, mapA, mapB, cnt, list_cap, S, sh);
      UPD_STAMP(8);
      alive = u_barrier(L, barriers, sh);
      UPD_STAMP(9);
    }
    if (alive) {
      if (!u_rank_few(L, sh)) u_rank_bins(L, sh);
      UPD_STAMP(10);
      if (tryR && (!wantB || sh.fast[1])) okR = u_rank_random(L, wantB, sh);
      UPD_STAMP(11);
    }
    // gradient-grown entries among the listed ones
    if (alive && tryB && sh.fast[1]) {
      const unsigned long long tau = sh.tau[1];
      for (int i = lane; i < cnt[1]; i += 32) {
        const unsigned long long v = S.list[i];
        if (v <= tau) {
          const uint32_t at = (uint32_t)v - lo_w * 32u;
          atomicOr(&S.grad[at >> 5], 1u << (at & 31u));
        }
      }
    }
  }
  const bool okA = tryA && sh.fast[0], okB = tryB && sh.fast[1];
  unsigned long long tauA = sh.tau[0], tauR = sh.rtau;
      UPD_STAMP(12);
  if (alive && wantA && !okA) alive = u_radix_select<U_PRUNE>(L, blk, lo_w, nloc, L.n_prune, barriers, gpass, S, sh, tauA);
  __syncthreads();
  // pruned entries (the few active entries of a word are neighbours in the value array)
  if (alive) {
    for (int i0 = 0; i0 < 2 * nloc; i0 += UT) {   // half a word per thread
      const int i = i0 + (int)threadIdx.x, li = i >> 1;
      const bool have = i < 2 * nloc;
      const uint32_t old = have && wantA ? S.old[li] : 0u;
      uint32_t m = old & ((i & 1) ? 0xFFFF0000u : 0xFFFFu), prn = 0;
      uint32_t pos = have ? (uint32_t)S.base[li] + ((i & 1) ? (uint32_t)__popc(old & 0xFFFFu) : 0u) : 0u;
      while (m) {
        const int b = __ffs(m) - 1;
        m &= m - 1;
        uint32_t key = u_prune_key(L, pos);
        const uint32_t slot = (lo_w + (uint32_t)li) * 32u + (uint32_t)b;
        if (L.lambda != 0.f) {
          const float g = fabsf(L.G[u_flat(L, lo_w + (uint32_t)li, b)]);
          key = __float_as_uint(__fadd_rn(__uint_as_float(key), __fmul_rn(L.lambda, g))) & 0x7FFFFFFFu;
        }
        // the bracket's threshold is a (key, position) pair, the radix select's a (key, slot) pair
        if ((((unsigned long long)key << 32) | (okA ? pos : slot)) <= tauA) prn |= 1u << b;
        ++pos;
      }
      __syncwarp();
      prn |= __shfl_xor_sync(0xffffffffu, prn, 1);
      if (have && !(i & 1)) S.prn[li] = prn;
    }
    __syncthreads();
  }
  if (alive && wantB && !okB) {
    unsigned long long tauB = 0;
    alive = u_radix_select<U_GRAD>(L, blk, lo_w, nloc, L.n_grad, barriers, gpass, S, sh, tauB);
    __syncthreads();
    if (alive) {
      for (int li = threadIdx.x >> 5; li < nloc; li += UW) {
        const uint32_t w = lo_w + (uint32_t)li, can = ~S.old[li] | (L.allow ? S.prn[li] : 0u);
        const bool cand = ((can >> lane) & 1u) && (int)((w % (uint32_t)L.wpr) * 32u) + lane < L.I;
        bool take = false;
        if (cand) take = (((unsigned long long)u_grad_key(L.G[u_flat(L, w, lane)]) << 32) | (w * 32u + (uint32_t)lane)) <= tauB;
        const unsigned g = __ballot_sync(0xffffffffu, take);
        if (lane == 0) S.grad[li] = g;
      }
      __syncthreads();
    }
  }
  const bool sweepR = wantR && !okR;
      UPD_STAMP(13);
  if (alive && sweepR) alive = u_radix_select<U_RAND>(L, blk, lo_w, nloc, L.n_rand, barriers, gpass, S, sh, tauR);
  __syncthreads();
  // new mask words and their population
  unsigned int pop = 0;
  if (alive) {
    for (int li = threadIdx.x; li < nloc; li += UT) {
      const uint32_t w = lo_w + (uint32_t)li, old = S.old[li], grad = S.grad[li];
      uint32_t m = 0, rnd = 0;
      if (wantR) {
        m = (sweepR ? ~old : S.hc[li]) & ~grad;
        const int left = L.I - (int)(w % (uint32_t)L.wpr) * 32;
        if (left < 32) m &= (1u << left) - 1u;
      }
      while (m) {
        const int b = __ffs(m) - 1;
        m &= m - 1;
        if (u_hash(L, w, b) <= tauR) rnd |= 1u << b;
      }
      const uint32_t nb = (old & ~S.prn[li]) | grad | rnd;
      S.hc[li] = nb;
      L.new_bits[w] = nb;
      pop += __popc(nb);
    }
    unsigned int before, dummy;
    u_scan2(pop, 0u, before, dummy, sh);
    if (threadIdx.x == UT - 1) L.bsums[blk] = (int32_t)(before + pop);
    UPD_STAMP(14);
    alive = u_barrier(L, barriers, sh);
    UPD_STAMP(15);
  }
  if (alive) {
    unsigned int off = 0, tot = 0;
    for (int j = threadIdx.x; j < L.blocks; j += UT) {
      const unsigned int x = (unsigned)__ldcg(L.bsums + j);
      tot += x;
      if (j < blk) off += x;
    }
    unsigned int eo, et;
    u_scan2(off, tot, eo, et, sh);
    if (threadIdx.x == UT - 1) { sh.below[0] = eo + off; sh.below[1] = et + tot; }
    __syncthreads();
    const unsigned int total = sh.below[1];
    const int chunk = (nloc + UT - 1) / UT, l0 = chunk * (int)threadIdx.x, l1 = l0 + chunk < nloc ? l0 + chunk : nloc;   // neighbouring words
    unsigned int x = 0;
    for (int li = l0; li < l1; ++li) x += __popc(S.hc[li]);
    unsigned int at, dummy;
    u_scan2(x, 0u, at, dummy, sh);
    at += sh.below[0];
    for (int li = l0; li < l1; ++li) {
      const uint32_t w = lo_w + (uint32_t)li, o = w / (uint32_t)L.wpr;
      S.prn[li] = at;
      L.new_wscan[w] = (int32_t)at;
      if (o * (uint32_t)L.wpr == w) L.new_row_ptr[o] = (int32_t)at;
      at += __popc(S.hc[li]);
    }
    if (blk == 0 && threadIdx.x == 0) {
      L.new_wscan[L.nwords] = (int32_t)total;
      L.new_row_ptr[L.O] = (int32_t)total;
    }
    __syncthreads();
    UPD_STAMP(16);
    if (L.bf16) u_fill<uint16_t>(L, lo_w, nloc, S);
    else u_fill<float>(L, lo_w, nloc, S);
      UPD_STAMP(17);
  }
  // the last block of the layer to get here leaves the scratch zero for the next launch
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    sh.r_n = atomicAdd(&L.ctr[C_EXIT], 1u) == (unsigned)L.blocks - 1u ? 1 : 0;
  }
  __syncthreads();
  if (sh.r_n) {
    for (int b = threadIdx.x; b < 5 * UBINS; b += UT) L.hist[b] = 0u;
    if (threadIdx.x < C_WORDS) L.ctr[threadIdx.x] = 0u;
  }
}

}  // namespace

mst_status_t mst_launch_fused_update(const UpdatePlan* plans, int n, int* taken, cudaStream_t s) {
  *taken = 0;
  static std::atomic<int> limits[64];   // dynamic shared memory a block can have, per device (0: not asked yet, -1: cannot run)
  int dev = 0;
  MST_CUDA_TRY(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) return MST_OK;
  int limit = limits[dev].load(std::memory_order_relaxed);
  if (limit == 0) {
    int coop = 0, optin = 0, occ = 0;
    cudaFuncAttributes fa;
    limit = -1;
    if (cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) == cudaSuccess && coop &&
        cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) == cudaSuccess &&
        cudaFuncGetAttributes(&fa, mg_update_kernel) == cudaSuccess) {
      const int most = optin - (int)fa.sharedSizeBytes;
      if (cudaFuncSetAttribute(mg_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most) == cudaSuccess &&
          cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, mg_update_kernel, UT, (size_t)most) == cudaSuccess && occ >= 1)
        limit = most;
    }
    limits[dev].store(limit, std::memory_order_relaxed);
  }
  if (limit < 0) return MST_OK;
  const int sms = mst_sm_count();

  // Blocks per layer: in proportion to the mask words, at least 64 words (2048 entries) per block, so that a barrier is not
  // waited for by blocks that have nothing to do.  A slice needs 20 bytes of shared memory per word; what is left holds the listed
  // entries, and at least one in eight of the slice's entries must fit, which is what the brackets of several layers need.
  // Layers are taken into the launch as long as that holds.
  UParams P = {};
  int words_cap = 0;
  for (int m = n < ULAYERS ? n : ULAYERS; m >= 1; --m) {
    int64_t total = 0;
    for (int i = 0; i < m; ++i) total += plans[i].L->nwords;
    int used = 0;
    words_cap = 0;
    for (int i = 0; i < m; ++i) {
      const int64_t nw = plans[i].L->nwords;
      int64_t b = nw * sms / (total > 0 ? total : 1);
      const int64_t most = (nw + 63) / 64, room = sms - used - (m - 1 - i);
      if (b > most) b = most;
      if (b > room) b = room;
      if (b < 1) b = 1;
      P.L[i].block0 = used;
      P.L[i].blocks = (int)b;
      used += (int)b;
      const int64_t per = (nw + b - 1) / b;
      if (per > words_cap) words_cap = per > (1 << 24) ? (1 << 24) : (int)per;
    }
    P.n = m;
    const int64_t left = (int64_t)limit - 20LL * words_cap;
    if (used <= sms && left >= 8 * 4096 && left / 8 >= 4LL * words_cap) break;
    P.n = 0;
  }
  if (P.n == 0) return MST_OK;
  int64_t cap = ((int64_t)limit - 20LL * words_cap) / 8;
  if (cap > 32LL * words_cap) cap = 32LL * words_cap;   // every entry of a slice
  if (cap < 4096) cap = 4096;                           // the samples are staged there
  P.words_cap = words_cap;
  P.list_cap = (int)cap;
  int grid = 0;
  for (int i = 0; i < P.n; ++i) {
    const UpdatePlan& pl = plans[i];
    mst_layer* L = pl.L;
    ULayer& u = P.L[i];
    u.old_bits = L->bits[pl.c]; u.old_wscan = L->wscan[pl.c]; u.vals = L->vals[pl.c];
    u.G = pl.P.G;
    u.stream = pl.P.stream; u.rand_lo = pl.rand_lo; u.rand_hi = pl.rand_hi; u.rand_bracket = pl.rand_bracket; u.rand_cap = L->rand_cap;
    u.new_bits = L->bits[pl.n]; u.new_wscan = L->wscan[pl.n]; u.new_row_ptr = L->row_ptr[pl.n];
    u.new_col = L->col_idx[pl.n]; u.new_vals = L->vals[pl.n];
    u.bsums = L->block_sums; u.flags = L->flags;
    u.hist = L->hist; u.ctr = L->upd_ctr; u.samples = L->upd_samples; u.bin_list = L->upd_list; u.rand_list = L->rand_list;
    u.n_prune = pl.n_prune; u.n_grad = pl.n_grad; u.n_rand = pl.n_rand;
    u.nnz = L->nnz; u.candidates = L->N - L->nnz;
    u.lambda = pl.P.lambda;
    u.nwords = (uint32_t)L->nwords;
    u.O = L->O; u.I = L->I; u.wpr = L->wpr; u.bf16 = L->dtype == MST_BF16; u.allow = pl.P.allow;
    grid += u.blocks;
    if (!L->scratch_clean) {
      MST_CUDA_TRY(cudaMemsetAsync(L->hist, 0, sizeof(unsigned int) * 5 * UBINS, s));
      MST_CUDA_TRY(cudaMemsetAsync(L->upd_ctr, 0, sizeof(unsigned int) * C_WORDS, s));
    }
    L->scratch_clean = 0;
  }
  const size_t smem = 8 * (size_t)P.list_cap + 20 * (size_t)P.words_cap;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(UT);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  // cooperative: the blocks of a layer wait for one another; overlapped: the kernel waits before its first access
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = mst_pdl_enabled() ? 2 : 1;
  MST_CUDA_TRY(cudaLaunchKernelEx(&cfg, mg_update_kernel, P));
  MST_COUNT_LAUNCH();
  for (int i = 0; i < P.n; ++i) {
    plans[i].L->scratch_clean = 1;
    plans[i].L->csc_valid = 0;
  }
  *taken = P.n;
  return MST_OK;
}

#ifdef MST_UPD_PROFILE
// (id, SM clock) pairs stamped by block 0 of the last update launch; returns the number of pairs
extern "C" int mst_update_profile(long long* out, int max_pairs) {
  long long h[64];
  int n = 0;
  if (cudaDeviceSynchronize() != cudaSuccess || cudaMemcpyFromSymbol(h, g_upd_stamps, sizeof(h)) != cudaSuccess ||
      cudaMemcpyFromSymbol(&n, g_upd_nstamps, sizeof(int)) != cudaSuccess)
    return -1;
  if (n > max_pairs) n = max_pairs;
  for (int i = 0; i < 2 * n; ++i) out[i] = h[i];
  return n;
}
#endif
