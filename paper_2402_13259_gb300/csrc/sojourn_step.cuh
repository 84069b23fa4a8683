// sojourn_step.cuh -- what the forms of the sojourn-time sampler (Sec. 6,
// Algorithm 4) share: a tagged customer's packed word and Lemma 3's
// conditional probability that its service continues.
#pragma once

#include <cstdint>

namespace eulernet {

// A customer's word: station << 32 | due step << 1 | setup pending.
constexpr unsigned long long kSojDone = 0xFFFFFFFFull << 32;

__device__ __forceinline__ unsigned long long soj_pack(int32_t station, int32_t due, bool setup) {
  return ((unsigned long long)(uint32_t)station << 32) | ((unsigned long long)(uint32_t)due << 1) |
         (setup ? 1ull : 0ull);
}

// b^k (k >= 0) by binary powering, multiplications in a fixed order.
__device__ __forceinline__ float soj_pow_int(float b, int32_t k) {
  float r = 1.0f;
  while (k > 0) {
    if (k & 1) r = r * b;
    b = b * b;
    k >>= 1;
  }
  return r;
}

// Lemma 3: P(the tagged customer's service continues through the step | the
// step's departure draw had input x and output d > 0, m servers).
__device__ __forceinline__ float soj_stay(int32_t x, int32_t d, int32_t m) {
  if (x <= m) return (float)(x - d) / (float)x;
  const float q = (float)(m - 1) / (float)m;
  if (x <= m + d) return soj_pow_int(q, x - m) * ((float)(x - d) / (float)m);
  return soj_pow_int(q, d);
}

}  // namespace eulernet
