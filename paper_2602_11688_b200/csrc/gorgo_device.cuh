// Device helpers shared by the kernels of libgorgo_b200.
#pragma once
#include "gorgo_internal.h"

namespace gorgo {

constexpr unsigned kFull = 0xFFFFFFFFu;

__device__ __forceinline__ double d_inf() { return __longlong_as_double(0x7FF0000000000000LL); }

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int d = 16; d > 0; d >>= 1) v += __shfl_xor_sync(kFull, v, d);
  return v;
}

// Is the touch `t` (of a request routed to replica `rep`) no longer its atom's latest touch there,
// looking at requests up to `r_now`?
__device__ __forceinline__ bool touch_is_stale(const Touch* touch, Touch t, const uint8_t* route_log,
                                               uint32_t rep, uint32_t r_now) {
  #pragma unroll 1
  while (t.next != kNone && t.next_req <= r_now) {
    if ((uint32_t)route_log[t.next_req] == rep) return true;
    t = touch[t.next];
  }
  return false;
}

__device__ __forceinline__ uint64_t mix64(uint64_t z) {  // splitmix64 finaliser
  z ^= z >> 30; z *= 0xbf58476d1ce4e5b9ULL;
  z ^= z >> 27; z *= 0x94d049bb133111ebULL;
  z ^= z >> 31;
  return z;
}

// First request x in [lo, hi] whose scaled arrival time is >= f; the caller knows that request
// hi qualifies.
__device__ __forceinline__ uint32_t first_arrival_at_or_after(const double* ts, double scale, double f,
                                                              uint32_t lo, uint32_t hi) {
  #pragma unroll 1
  while (lo < hi) {                                       // at most 32 rounds
    const uint32_t mid = lo + ((hi - lo) >> 1);
    if (__dmul_rn(scale, ts[mid]) >= f) hi = mid; else lo = mid + 1;
  }
  return lo;
}

}  // namespace gorgo
