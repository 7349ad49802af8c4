// Forward copy of idle user rows, shared by the SGD kernels.
#pragma once

#include "internal.h"
#include "ptx.cuh"

namespace esspt {

// Forward copy of the users with no entry in minibatch b: the row of version
// c-1 becomes that of version c.  One warp per 32 consecutive users: their
// entry counts come from two coalesced offset loads, and each row group
// copies the idle ones among its 32/kGpw, up to 8 slices per lane in flight.
// A row unchanged over the last s+2 clocks is skipped: the ring slot of
// version c last held version c-(s+2), which is already its value.
template <int G, int NV>
__device__ __forceinline__ void copy_idle_users(const SgdArgs& a, int64_t warp, int64_t nwarps, int lane) {
  constexpr int kGpw = 32 / G;                     // rows side by side in a warp
  constexpr int kRows = G;                         // rows per group and unit
  constexpr int kBatch = kRows < 8 / NV ? kRows : 8 / NV;  // rows in flight per group
  const int glane = lane & (G - 1), grp = lane / G;
  const int32_t K4 = a.K >> 2;
  const int64_t slot4 = a.n_rows * K4;
  float4* ring4 = reinterpret_cast<float4*>(a.ring) + glane;
  const float4* base4 = ring4 + (int64_t)a.slot_base * slot4;
  float4* out4 = ring4 + (int64_t)a.slot_out * slot4;
  const uint64_t pol = policy_evict_first();
  const bool may_skip = a.clock > a.copy_all_until;
  for (int64_t u0 = warp * 32; u0 < a.n_users; u0 += nwarps * 32) {
    const int64_t u = u0 + lane;
    bool idle = false;
    if (u < a.n_users) {
      idle = __ldg(a.uoff + u + 1) == __ldg(a.uoff + u);
      if (idle && may_skip && a.clock - ld_stream_i32(a.chg + u, pol) >= a.nslots) idle = false;
    }
    const unsigned mask = __ballot_sync(0xffffffffu, idle);
    if (mask == 0u) continue;
#pragma unroll 1
    for (int q0 = 0; q0 < kRows; q0 += kBatch) {
      float4 v[kBatch][NV];
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int r = (q0 + q) * kGpw + grp;
        const bool on = (mask >> r) & 1u;
#pragma unroll
        for (int t = 0; t < NV; ++t)
          v[q][t] = ld_stream_if(base4 + (u0 + r) * K4 + t * G, pol, on && (t < NV - 1 || glane + t * G < K4));
      }
#pragma unroll
      for (int q = 0; q < kBatch; ++q) {
        const int r = (q0 + q) * kGpw + grp;
        const bool on = (mask >> r) & 1u;
#pragma unroll
        for (int t = 0; t < NV; ++t)
          st_stream_if(out4 + (u0 + r) * K4 + t * G, v[q][t], pol, on && (t < NV - 1 || glane + t * G < K4));
      }
    }
  }
}

}  // namespace esspt
