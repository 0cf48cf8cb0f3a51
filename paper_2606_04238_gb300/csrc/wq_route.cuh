// wq_route.cuh -- a token's experts by router logit, one warp: the larger logit
// first, the lower expert index among equal ones.  A NaN ranks by its sign, above
// every number or below, so the order is total.  Shared by the routing launches of
// the slots and of the grouped experts, and by the gate/up launch over the slots,
// which finds its own expert so that it need not wait for the former.
#pragma once

#include <cstdint>

namespace wq {

constexpr int kMoeMaxExperts = 256;

// Lane l holds experts l, l + 32, .. as integers in the logits' order; taken
// ones are marked by clearing their bit.
struct RouteKeys {
  uint32_t k[kMoeMaxExperts / 32];
  uint32_t live;
};

__device__ __forceinline__ void route_load(RouteKeys &s, const float *logits, int E, int lane) {
  s.live = 0u;
#pragma unroll
  for (int i = 0; i < kMoeMaxExperts / 32; ++i) {
    const int e = lane + 32 * i;
    s.k[i] = 0u;
    if (e < E) {
      const float v = __ldcg(logits + e);
      const uint32_t u = v == 0.f ? 0u : __float_as_uint(v);  // -0 equals +0
      s.k[i] = u & 0x80000000u ? ~u : u | 0x80000000u;
      s.live |= 1u << i;
    }
  }
}

// The next expert (the same in every lane) and its logit.
__device__ __forceinline__ int route_next(RouteKeys &s, int lane, float &logit) {
  uint32_t best = 0u;
#pragma unroll
  for (int i = 0; i < kMoeMaxExperts / 32; ++i)
    if ((s.live >> i) & 1u) best = max(best, s.k[i]);
  best = __reduce_max_sync(0xffffffffu, best);
  uint32_t e = 0xffffffffu;
#pragma unroll
  for (int i = kMoeMaxExperts / 32 - 1; i >= 0; --i)
    if (((s.live >> i) & 1u) && s.k[i] == best) e = lane + 32 * i;
  e = __reduce_min_sync(0xffffffffu, e);
  if ((int)(e & 31u) == lane) s.live &= ~(1u << (e >> 5));
  logit = __uint_as_float(best & 0x80000000u ? best & 0x7fffffffu : ~best);
  return (int)e;
}

}  // namespace wq
