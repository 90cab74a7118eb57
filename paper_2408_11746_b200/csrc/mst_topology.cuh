// Shared by the forms of the topology update: selection parameters, the random-growth generator, one layer's plan.
#pragma once
#include <stdint.h>

#include "mst_internal.cuh"

struct SelParams {
  const uint32_t* old_bits;
  const int32_t* old_wscan;
  const void* vals;
  int bf16;
  const float* G;
  const uint32_t* pruned_bits;
  const uint32_t* grad_bits;
  int O, I, wpr, allow;
  int aligned;   // I % 32 == 0
  int low_zero;  // low key bits known to be zero in the prune keys (16 for bf16 values)
  float lambda;  // MEST prune key |w| + lambda |g| when non-zero
  int64_t nwords;
  unsigned long long stream;
};

// SplitMix64 output function (Steele, Lea, Flood 2014).  A bijection, and the generator's states of two entries differ, so
// no two entries of a layer have equal hash keys.
__host__ __device__ __forceinline__ unsigned long long sm64_mix(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
// the same without the last step, which changes only the lowest bit of the high word
__host__ __device__ __forceinline__ unsigned long long sm64_mix_top(unsigned long long z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  return (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
}
constexpr unsigned long long SM64_GAMMA = 0x9E3779B97F4A7C15ULL;

// One layer's update, planned on the host: counts, selection parameters, which buffer set is built.
struct UpdatePlan {
  mst_layer* L;
  int64_t n_prune, n_rand, n_grad, target;
  int c, n;  // live set, set being built
  SelParams P;
  unsigned long long rand_lo, rand_hi;  // bracket of the random growth's threshold (rand_bracket = 0: none planned)
  int rand_bracket;
};

// One cooperative launch for the updates of several layers (mst_update_fused.cu).  *taken: how many of the n plans, from the
// first on, the launch has taken (0: the first one does not fit and needs the kernel-per-phase form).
mst_status_t mst_launch_fused_update(const UpdatePlan* plans, int n, int* taken, cudaStream_t s);
