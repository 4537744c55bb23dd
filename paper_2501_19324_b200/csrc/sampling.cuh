// What the kernels that sample share: scores packed for atomic maxima, the quick form of the Gumbel noise and the margins that go with it.
#pragma once

#include "common.cuh"

namespace rsd {

__device__ __forceinline__ void better(float& bs, int& bi, float s, int i) {
  if (s > bs || (s == bs && i < bi)) { bs = s; bi = i; }
}

// Order-preserving image of a score; 0 is below every number's.
__device__ __forceinline__ uint32_t score_key(float sc) {
  const uint32_t b = __float_as_uint(sc);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// (score, id) packed so that an unsigned 64-bit maximum picks the highest score and, among equal
// scores, the lowest id: high word = order-preserving image of the float, low word = ~id.
__device__ __forceinline__ unsigned long long pack_best(float sc, int id) {
  return ((unsigned long long)score_key(sc) << 32) | (uint32_t)(0xFFFFFFFFu - (uint32_t)id);
}

__device__ __forceinline__ float unpack_score(unsigned long long packed) {
  const uint32_t key = (uint32_t)(packed >> 32);
  return __uint_as_float((key & 0x80000000u) ? key ^ 0x80000000u : ~key);
}

constexpr float kScoreMargin = 1e-3f;       // the fast score errs by less than 1e-4 (see fast_gumbel)
constexpr float kNoiseMax = 17.f;           // the noise lies below 16.64

// -log(-log u) for u = (2k + 1) / 2^24.  Near 1, where the large values come from, -log u is its series in 1 - u (exact
// in fp32; 1 - u < 2^-6: three terms err by 1e-6 relative); elsewhere __logf errs by 2^-21.4 on -log u > 2^-6, that is
// 2.3e-5 relative, and so much in the outer logarithm, whose own error is 3 ulp of at most 17.
__device__ __forceinline__ float fast_gumbel(float u) {
  const float d = 1.f - u;
  const float y = d < 0.015625f ? d * (1.f + d * (0.5f + d * 0.33333333f)) : -__logf(u);
  return -__logf(y);
}

// What still can win against a best score of `run`.
__device__ __forceinline__ float score_needed(float run) {
  return run == INFINITY ? run : run - (kScoreMargin + fabsf(run) * 1e-6f);
}

}  // namespace rsd
