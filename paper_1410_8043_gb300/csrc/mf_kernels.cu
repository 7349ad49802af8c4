// Matrix-factorisation SGD on the version ring (Sec. 3.1 updates under the
// SSP / ESSP read schedule).  One clock is:
//   sgd_stream_kernel   every user with entries (its row of version c,
//                       written once), every chunk of a very active one, and
//                       the rows of users without entries, carried from
//                       version c-1 to version c unless the ring already
//                       holds them;
//   heavy_merge_kernel  rows of the very active users (if any);
//   item_merge_kernel   the Clock() merge of the item rows.
// Item-row (and heavy-user) deltas are summed, unscaled, into zero-initialised
// replica rows so that popular rows spread their fp32 reductions over many
// L2 addresses; the merges apply eta, the hot-row scale and the sum of the
// replicas, then clear them for the next clock.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"
#include "schedule.cuh"

namespace esspt {

namespace {

// Sum over the G lanes of a row group (G a power of two, <= 32).
template <int G>
__device__ __forceinline__ float group_sum(float x, unsigned mask) {
#pragma unroll
  for (int off = G / 2; off > 0; off >>= 1) x += __shfl_xor_sync(mask, x, off, G);
  return x;
}

__device__ __forceinline__ float4 f4_zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

__device__ __forceinline__ float dot4(float4 a, float4 b) { return a.x * b.x + a.y * b.y + a.z * b.z + a.w * b.w; }

__device__ __forceinline__ float4 f4_axpy(float s, float4 x, float4 y) {  // y + s x
  return make_float4(y.x + s * x.x, y.y + s * x.y, y.z + s * x.z, y.w + s * x.w);
}

// Scale of a row's summed update under the hot-row step cap.
__device__ __forceinline__ float cap_scale(int32_t cap, int32_t n) {
  return (cap > 0 && n > cap) ? (float)cap / (float)n : 1.f;
}

// cap / n for a row past the cap, out of line: the rare case stays off the
// common path.
__device__ __noinline__ float capped_scale(int32_t cap, int32_t n) { return (float)cap / (float)n; }

__device__ __forceinline__ float4 f4_add(float4 a, float4 b) {
  return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// Sum of n replica slices p[0], p[stride], ..., each cleared after reading;
// eight independent loads in flight per lane.
__device__ __forceinline__ float4 sum_and_clear(float4* p, int32_t n, int32_t stride) {
  float4 acc = f4_zero();
  int32_t r = 0;
  for (; r + 8 <= n; r += 8) {
    float4 x[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) x[k] = p[(int64_t)(r + k) * stride];
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      p[(int64_t)(r + k) * stride] = f4_zero();
      acc = f4_add(acc, x[k]);
    }
  }
  for (; r < n; ++r) {
    acc = f4_add(acc, p[(int64_t)r * stride]);
    p[(int64_t)r * stride] = f4_zero();
  }
  return acc;
}

__device__ __forceinline__ void flush_loss(double* out, float v, int lane) {
  if (out == nullptr) return;
  double x = (double)v;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  if (lane == 0 && x != 0.0) atomicAdd(out, x);
}

}  // namespace

constexpr int kStreamWarps = 4;   // warps per block

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

// One clock of MF-SGD over minibatch b.  The work list holds one item per user
// with 1..kHeavy entries and one per 64-entry chunk of a heavy user, sorted by
// length within tiles of consecutive users.  A warp walks one contiguous range
// of items in rounds of 32/G: each row group of G lanes (NV float4 slices of a
// row per lane, slice glane + t G on lane glane) takes one item, and the groups
// step through their items' entries together, one entry per group and step:
//   e = D - L.R,  gL += e R,  dR[dst] += e L - lambda R
// At the end of a round every group closes its item: a user's row of version c
// = base + eta s (gL - n lambda L), written once; a chunk's partial sum goes,
// unscaled, into its replica row of dL.
//
// The work is bound by issue slots, not by memory (the kernels this replaces
// took 80..92% of their time with the gathers served by L1 and the reductions
// left out), so it is built to issue little: the 32/G groups share every
// instruction, rounds included, since the items of a round have (nearly) one
// length; packed fp32 pairs (fma.rn.f32x2); one broadcast shared-memory read
// for an entry's item, replica row, value and count; constant offsets from one
// pointer per row; log2 G shuffles per step for 32/G dot products.
// In flight per group: the next entry's item row (registers), the user rows
// and first window of the next item (cp.async; every lane copies and reads its
// own slices only), the item's next window.
template <int G, int NV, int MINB, int HOT>
__global__ void __launch_bounds__(kStreamWarps * 32, MINB) sgd_stream_kernel(StreamArgs c) {
  constexpr int kGpw = 32 / G;
  constexpr int kWindow = G < 8 ? G : 8;       // records per window of a row group
  constexpr int kRecs = kGpw * (kWindow + 1);  // per window buffer: groups fall on different banks
  __shared__ __align__(16) float4 stageL[kStreamWarps][NV][32];
  __shared__ __align__(16) float4 stageB[kStreamWarps][2][NV][32];
  // window buffers: the first windows of this round and the next, then two for later windows
  __shared__ __align__(16) int4 recs[kStreamWarps][4][kRecs];
  __shared__ __align__(16) int4 metas[kStreamWarps][2][kGpw];
  // per warp and lane: the summed updates of the minibatch's hot items
  __shared__ __align__(16) float4 hot[kStreamWarps][HOT > 0 ? HOT : 1][NV][HOT > 0 ? 32 : 1];
  // row mode (the launch asks for it then): ring row of each record's item
  extern __shared__ int32_t rows_dyn[];
  const SgdArgs& a = c.a;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  int32_t* rows = rows_dyn + wib * 4 * kRecs;
  const int glane = lane & (G - 1), grp = lane / G;
  const int32_t K4 = a.K >> 2;
  const bool last_on = glane + (NV - 1) * G < K4;  // the lane's last slice lies inside the row
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  float loss = 0.f;

  // Half of the warps copy idle rows first, the others last: the copy's DRAM
  // traffic runs beside the other warps' arithmetic.
  if (warp & 1) copy_idle_users<G, NV>(a, warp, nwarps, lane);

  int32_t xa = 0, xb = 0;
  if (warp < c.n_warps) {
    xa = __ldg(c.part + warp);
    xb = __ldg(c.part + warp + 1);
  }
  if (xa < xb) {
    const int64_t slot4 = a.n_rows * K4;
    float4* ring4 = reinterpret_cast<float4*>(a.ring) + glane;
    const uint64_t pol = policy_evict_first();
    auto load_item = [&](int32_t r0) {  // the group's item of the round that starts at item r0
      const int32_t x = r0 + grp;
      return x < xb ? __ldg(c.items + x) : make_int4(0, 0, -2, 0);
    };
    // Records [at, at + n) of the stream, n <= kWindow, into window buffer w.
    auto fetch_window = [&](int w, int32_t at, int32_t n) {
#pragma unroll
      for (int l = glane; l < kWindow; l += G) {
        cp_async16_hint_if(&recs[wib][w][grp * (kWindow + 1) + l], c.rec + at + l, l < n, pol);
        if (a.row_mode) cp_async4_if(rows + w * kRecs + grp * (kWindow + 1) + l, a.rec_row + at + l, l < n);
      }
    };
    // Rows, first window and metadata of the next round's item, in half sb of
    // the double buffers.
    auto stage = [&](const int4& it, int sb) {
      const int32_t n = it.w >> 16;
      const int32_t vs = a.row_mode ? __ldg(a.user_slot + it.x) : __ldg(a.vslot + (it.w & 0xffff));
      const float4* pv = ring4 + vs * slot4 + (int64_t)it.x * K4;
      const float4* pb = ring4 + a.slot_base * slot4 + (int64_t)it.x * K4;
      const bool bon = it.z == -1 && vs != a.slot_base;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const bool in = k < NV - 1 || last_on;
        cp_async16_hint_if(&stageL[wib][k][lane], pv + k * G, n > 0 && in, pol);
        cp_async16_hint_if(&stageB[wib][sb][k][lane], pb + k * G, bon && in, pol);
      }
      fetch_window(sb, it.y, n);
      if (glane == 0) metas[wib][sb][grp] = make_int4(it.x, it.y, it.z, vs << 7 | n);
    };

#pragma unroll
    for (int k = 0; k < NV; ++k) stageL[wib][k][lane] = f4_zero();  // slices past the row end stay zero
#pragma unroll
    for (int h = 0; h < HOT; ++h)
#pragma unroll
      for (int k = 0; k < NV; ++k) hot[wib][h][k][lane] = f4_zero();
    int32_t xr = xa;  // first item of the current round
    int4 far = load_item(xr);
    stage(far, 0);
    cp_async_commit();
    far = load_item(xr + kGpw);
    cp_async_wait_all();
    __syncwarp();

    // Current round.
    f2x2 L[NV], gL[NV];
    int32_t cur_u = 0, cur_beg = 0, cur_z = 0, cur_n = 0, cur_vs = 0, steps = 0;
    const float4* cur_R = ring4;
    int sb = 0;                 // the round's half of the double buffers
    int win = 0;                // window buffer of entry i
    auto item_rows = [&](int32_t vs) -> const float4* {
      return a.row_mode ? ring4 : ring4 + vs * slot4 + (int64_t)a.n_users * K4;
    };
    auto open_round = [&]() {
      const int4 m = metas[wib][sb][grp];
      cur_u = m.x;
      cur_beg = m.y;
      cur_z = m.z;
      cur_n = m.w & 127;
      cur_vs = m.w >> 7;
      cur_R = item_rows(cur_vs);
      steps = __reduce_max_sync(0xffffffffu, cur_n);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        L[k] = lds_f2x2(&stageL[wib][k][lane]);
        gL[k] = f2x2{0ull, 0ull};
      }
      win = sb;
      if (xr + kGpw < xb) stage(far, sb ^ 1);
      if (steps > kWindow) fetch_window(2, cur_beg + kWindow, cur_n - kWindow);
      cp_async_commit();
      far = load_item(xr + 2 * kGpw);
    };
    open_round();

    f2x2 Ra[NV], Rb[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) Ra[k] = Rb[k] = f2x2{0ull, 0ull};
    int4 ra = recs[wib][0][grp * (kWindow + 1)], rb;
    if (cur_n > 0) {
      const float4* row = cur_R + (int64_t)(a.row_mode ? rows[grp * (kWindow + 1)] : ra.x) * K4;
#pragma unroll
      for (int k = 0; k < NV; ++k) ldg_f2x2_if(Ra[k], row + k * G, k < NV - 1 || last_on);
    }

    // Step i of the round: the group's entry i (record rc, item row Rc), and
    // the gather of the entry after it, of this round or the next, into Rn.
    const u64 nlam = pack2(-a.lambda, -a.lambda);
    int32_t i = 0;
    auto step = [&](const int4& rc, int4& rn, const f2x2(&Rc)[NV], f2x2(&Rn)[NV]) {
      const bool last = i + 1 == steps;
      const float4* base = cur_R;
      int at = grp * (kWindow + 1);
      bool more;
      if (last) {  // the next round's first entries
        cp_async_wait_all();
        __syncwarp();
        win = sb ^ 1;
        const int32_t w = metas[wib][sb ^ 1][grp].w;
        more = xr + kGpw < xb && (w & 127) > 0;
        base = item_rows(w >> 7);
      } else {
        const int o = (i + 1) & (kWindow - 1);
        if (o == 0) {  // the item's next window
          cp_async_wait_all();
          __syncwarp();
          const int32_t w = (i + 1) / kWindow;
          win = 2 + ((w - 1) & 1);
          if (steps > i + 1 + kWindow) {
            fetch_window(2 + (w & 1), cur_beg + i + 1 + kWindow, cur_n - (i + 1 + kWindow));
            cp_async_commit();
          }
        }
        at += o;
        more = i + 1 < cur_n;
      }
      rn = recs[wib][win][at];
      {
        const float4* row = base + (int64_t)(a.row_mode ? rows[win * kRecs + at] : rn.x) * K4;
#pragma unroll
        for (int k = 0; k < NV; ++k) ldg_f2x2_if(Rn[k], row + k * G, more && (k < NV - 1 || last_on));
      }
      u64 p = mul2(L[0].lo, Rc[0].lo);
      p = fma2(L[0].hi, Rc[0].hi, p);
#pragma unroll
      for (int k = 1; k < NV; ++k) {
        p = fma2(L[k].lo, Rc[k].lo, p);
        p = fma2(L[k].hi, Rc[k].hi, p);
      }
      float dot = sum2(p);
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
      if (i < cur_n) {
        const float e = __int_as_float(rc.z) - dot;
        loss += e * e;
        const u64 ee = pack2(e, e);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          gL[k].lo = fma2(ee, Rc[k].lo, gL[k].lo);
          gL[k].hi = fma2(ee, Rc[k].hi, gL[k].hi);
        }
        if (HOT > 0 && rc.y < 0) {
#pragma unroll
          for (int k = 0; k < NV; ++k) {
            float4* h = &hot[wib][-1 - rc.y][k][lane];
            const f2x2 v = lds_f2x2(h);
            sts_f2x2(h, add2(v.lo, fma2(ee, L[k].lo, mul2(nlam, Rc[k].lo))),
                     add2(v.hi, fma2(ee, L[k].hi, mul2(nlam, Rc[k].hi))));
          }
        } else {
          float4* out = reinterpret_cast<float4*>(a.dR) + glane + (int64_t)rc.y * a.dR_ld;
#pragma unroll
          for (int k = 0; k < NV; ++k)
            red_add_f2x2_if(out + k * G, fma2(ee, L[k].lo, mul2(nlam, Rc[k].lo)),
                            fma2(ee, L[k].hi, mul2(nlam, Rc[k].hi)), k < NV - 1 || last_on);
        }
      }
    };
    auto close_round = [&]() {
      const float nl = -a.lambda * (float)cur_n;
      const u64 nl2 = pack2(nl, nl);
      if (cur_z == -1) {
        float sc = a.eta;
        if (a.cap > 0 && cur_n > a.cap) sc = a.eta * capped_scale(a.cap, cur_n);
        const u64 sc2 = pack2(sc, sc);
        float4* o = ring4 + a.slot_out * slot4 + (int64_t)cur_u * K4;
        const bool same = cur_vs == a.slot_base;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          f2x2 b = L[k];
          if (!same) b = lds_f2x2(&stageB[wib][sb][k][lane]);
          st_stream_f2x2_if(o + k * G, fma2(sc2, fma2(nl2, L[k].lo, gL[k].lo), b.lo),
                            fma2(sc2, fma2(nl2, L[k].hi, gL[k].hi), b.hi), pol, k < NV - 1 || last_on);
        }
        if (glane == 0) a.chg[cur_u] = a.clock;
      } else if (cur_z >= 0) {
        float4* o = reinterpret_cast<float4*>(c.dL) + (int64_t)cur_z * K4 + glane;
#pragma unroll
        for (int k = 0; k < NV; ++k)
          red_add_f2x2_if(o + k * G, fma2(nl2, L[k].lo, gL[k].lo), fma2(nl2, L[k].hi, gL[k].hi),
                          k < NV - 1 || last_on);
      }
    };
    // After each step: at the round's end close it and open the next.
    auto next = [&]() -> bool {
      if (++i < steps) return true;
      close_round();
      xr += kGpw;
      if (xr >= xb) return false;
      sb ^= 1;
      i = 0;
      open_round();
      return true;
    };
    for (;;) {
      step(ra, rb, Ra, Rb);
      if (!next()) break;
      step(rb, ra, Rb, Ra);
      if (!next()) break;
    }
    cp_async_wait_all();
    // Hot items: the groups' sums, added once into a replica row of the item
    // (the warp index picks among its replicas).
#pragma unroll
    for (int h = 0; h < HOT; ++h) {
      const int32_t j = __ldg(a.hot_item + h);
      if (j < 0) continue;
      const int32_t e0 = __ldg(a.item_rep + j), e1 = __ldg(a.item_rep + j + 1);
      const int32_t rep = (int32_t)(warp & (int64_t)(e1 - e0));  // replicas are a power of two
      const int64_t row = rep == 0 ? (int64_t)j : a.n_rows - a.n_users + e0 + rep - 1;
      float4* out = reinterpret_cast<float4*>(a.dR) + row * a.dR_ld + glane;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        float4 v = hot[wib][h][k][lane];
#pragma unroll
        for (int off = G; off < 32; off <<= 1) {
          v.x += __shfl_xor_sync(0xffffffffu, v.x, off);
          v.y += __shfl_xor_sync(0xffffffffu, v.y, off);
          v.z += __shfl_xor_sync(0xffffffffu, v.z, off);
          v.w += __shfl_xor_sync(0xffffffffu, v.w, off);
        }
        if (grp == 0 && (k < NV - 1 || last_on)) atomicAdd(out + k * G, v);
      }
    }
  }
  if (!(warp & 1)) copy_idle_users<G, NV>(a, warp, nwarps, lane);
  flush_loss(a.sq_loss, glane == 0 ? loss : 0.f, lane);
}

// Row-granular SSP (Sec. 4 client cache, a clock c_param per cached row): for
// every work item, refresh its user's row and its records' item rows in the
// cache of the reading worker.  Eight lanes per item, one record per lane and
// pass.  All lanes that refresh one (worker, row) in a clock write the same
// value, c-1, so the races are benign and every read of the row in the clock
// sees one version.
__global__ void __launch_bounds__(256) row_refresh_kernel(RowRefreshArgs a) {
  const int32_t lo = a.c - 1 - a.s;
  const int l = threadIdx.x & 7;
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t x = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; x < a.n_items; x += stride) {
    const int4 it = __ldg(a.items + x);
    int32_t* V = a.rowver + (int64_t)(it.w & 0xffff) * a.n_rows;
    const int32_t n = it.w >> 16;
    if (l == 0) {
      int32_t v = V[it.x];
      if (v < 0 || v < lo) {
        v = a.c - 1;
        V[it.x] = v;
      }
      a.user_slot[it.x] = v % a.nslots;
    }
    for (int32_t k = l; k < n; k += 8) {
      const int64_t r = (int64_t)a.n_users + __ldg(&a.rec[it.y + k].x);
      int32_t v = V[r];
      if (v < 0 || v < lo) {
        v = a.c - 1;
        V[r] = v;
      }
      a.rec_row[it.y + k] = (int32_t)((int64_t)(v % a.nslots) * a.n_rows + r);
    }
  }
}

// Heavy user rows: L^c = L^base + eta s sum of the user's replica rows (row u
// of dL, then rows hv.y .. hv.y + hv.z - 2); the replicas are cleared for the
// next clock.  One warp per heavy user.
__global__ void __launch_bounds__(256) heavy_merge_kernel(HeavyMergeArgs a) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int32_t K4 = a.K >> 2;
  const int64_t slot4 = a.n_rows * K4;
  float4* ring4 = reinterpret_cast<float4*>(a.ring);
  float4* dL4 = reinterpret_cast<float4*>(a.dL);
  for (int64_t h = warp; h < a.n_heavy; h += nwarps) {
    const int4 hv = a.heavy[h];
    const float sc = a.eta * cap_scale(a.cap, hv.w);
    for (int32_t q = lane; q < K4; q += 32) {
      float4* p0 = dL4 + (int64_t)hv.x * K4 + q;
      float4 acc = *p0;
      *p0 = f4_zero();
      acc = f4_add(acc, sum_and_clear(dL4 + (int64_t)hv.y * K4 + q, hv.z - 1, K4));
      const float4 b = ring4[(int64_t)a.slot_base * slot4 + (int64_t)hv.x * K4 + q];
      ring4[(int64_t)a.slot_out * slot4 + (int64_t)hv.x * K4 + q] = f4_axpy(sc, acc, b);
    }
    if (lane == 0) a.chg[hv.x] = a.clock;
  }
}

// Clock() merge of the item rows (Sec. 2.1 additive updates, Sec. 4 server
// clock): R^c_j = R^base_j + eta s_j sum of j's replica rows; replicas
// cleared.  Each thread merges U (item, float4 slice) pairs.  Replica 0 of
// item j is row j of dR, so the common single-replica item needs no index
// load before its data loads: every load of a thread is issued at once.  With do_schedule the
// first P threads also compute the next clock's read versions (the SGD
// kernels of this clock, the only readers of v, have finished).
template <int U>  // (item, slice) pairs per thread per round, the loads of all in flight
__global__ void __launch_bounds__(256) item_merge_kernel(ItemMergeArgs a) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  if (a.do_schedule)
    for (int64_t p = tid; p < a.sched.P; p += nth) schedule_worker(a.sched, (int32_t)p);
  const int32_t K4 = a.K >> 2;
  const int64_t slot4 = a.n_rows * K4;
  float4* ring4 = reinterpret_cast<float4*>(a.ring);
  float4* dR4 = reinterpret_cast<float4*>(a.dR);
  // n_items * K/4 < 2^31 (checked at load), so the (item, slice) split is a
  // 32-bit division
  const int64_t total = (int64_t)a.n_items * K4;
  for (int64_t x0 = tid; x0 < total; x0 += U * nth) {
    float4 first[U], base[U];
    int32_t e0[U], e1[U], cnt[U];
    int64_t row[U], dofs[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const int64_t x = min(x0 + k * nth, total - 1);
      const uint32_t j = (uint32_t)x / (uint32_t)K4;
      const int32_t q = (int32_t)((uint32_t)x - j * (uint32_t)K4);
      row[k] = ((int64_t)a.n_users + j) * K4 + q;
      dofs[k] = (int64_t)j * a.dR_ld + q;
      first[k] = dR4[dofs[k]];
      base[k] = ring4[(int64_t)a.slot_base * slot4 + row[k]];
      e0[k] = __ldg(a.item_rep + j);
      e1[k] = __ldg(a.item_rep + j + 1);
      cnt[k] = __ldg(a.item_cnt + j);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      if (x0 + k * nth >= total) break;
      dR4[dofs[k]] = f4_zero();
      float4 acc = first[k];
      if (e1[k] > e0[k]) {
        const int32_t q = (int32_t)(dofs[k] % a.dR_ld);
        acc = f4_add(acc, sum_and_clear(dR4 + ((int64_t)a.n_items + e0[k]) * a.dR_ld + q, e1[k] - e0[k], a.dR_ld));
      }
      const float sc = a.eta * cap_scale(a.cap, cnt[k]);
      ring4[(int64_t)a.slot_out * slot4 + row[k]] = f4_axpy(sc, acc, base[k]);
    }
  }
}

namespace {

int sm_count() {
  static int sms = 0;
  if (sms == 0) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (sms <= 0) sms = 148;
  }
  return sms;
}

int grid_for(int64_t work_items, int64_t per_block, int max_per_sm) {
  const int64_t want = (work_items + per_block - 1) / per_block;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sm_count() * max_per_sm));
}

// Row-group shape for K: G lanes per row (a power of two) and NV float4 slices
// per lane, G (NV - 1) < K/4 <= G NV, and the blocks per SM the kernel is
// compiled for.  Eight lanes read 128 consecutive bytes per load, a whole
// line; wider groups only where NV = 4 slices per lane do not hold the row.
// Blocks per SM: as many as spill (next to) nothing; on the 300k x 40k, K=48
// case 6 blocks take 122 us, 7 blocks 128, 8 blocks (64 registers, spills)
// 213; 5 blocks with rows staged two rounds ahead 131; on 480k x 18k, K=100
// 4 blocks 443 us, 5 blocks (spills) 785, 3 blocks 525 (before the wider
// replica rows, where 4 blocks took 508).
template <int G_, int NV_, int MINB_, int HOT_ = 0>
struct StreamShape {
  static constexpr int G = G_, NV = NV_, MINB = MINB_, HOT = HOT_, GPW = 32 / G_;
};
template <typename F>
auto dispatch_stream(int32_t K, F&& f) {
  const int32_t K4 = K / 4;
  if (K4 <= 4) return f(StreamShape<4, 1, 8>{});
  if (K4 <= 8) return f(StreamShape<8, 1, 7>{});
  if (K4 <= 16) return f(StreamShape<8, 2, 6, kHot>{});
  if (K4 <= 24) return f(StreamShape<8, 3, 4>{});
  if (K4 <= 32) return f(StreamShape<8, 4, 4>{});
  if (K4 <= 48) return f(StreamShape<16, 3, 4>{});
  if (K4 <= 64) return f(StreamShape<16, 4, 4>{});
  if (K4 <= 96) return f(StreamShape<32, 3, 4>{});
  return f(StreamShape<32, 4, 4>{});
}

}  // namespace

int64_t stream_max_warps(int32_t K) {
  return dispatch_stream(K, [](auto s) { return (int64_t)sm_count() * s.MINB * kStreamWarps; });
}

int stream_groups_per_warp(int32_t K) {
  return dispatch_stream(K, [](auto s) { return s.GPW; });
}

cudaError_t launch_sgd_stream(const StreamArgs& c, cudaStream_t st) {
  return dispatch_stream(c.a.K, [&](auto s) {
    using S = decltype(s);
    const auto kernel = sgd_stream_kernel<S::G, S::NV, S::MINB, S::HOT>;
    static bool configured = false;
    if (!configured) {
      // The smallest shared-memory carveout that holds the resident blocks'
      // staging buffers: the rest of the SM's memory is L1, which keeps the
      // popular item rows.
      cudaFuncAttributes at{};
      cudaError_t e = cudaFuncGetAttributes(&at, kernel);
      if (e != cudaSuccess) return e;
      const int64_t need = ((int64_t)at.sharedSizeBytes + 1024) * S::MINB, all = 228 * 1024;
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                               (int)std::min<int64_t>(100, (need * 100 + all - 1) / all));
      if (e != cudaSuccess) return e;
      configured = true;
    }
    // Warps for the work list, and one per 32 users for the forward copy, up
    // to one resident wave.
    const int64_t warps = std::max<int64_t>(c.n_warps, (c.a.n_users + 31) / 32);
    const int win = S::G < 8 ? S::G : 8;
    const size_t rows = c.a.row_mode ? sizeof(int32_t) * kStreamWarps * 4 * S::GPW * (win + 1) : 0;
    kernel<<<grid_for(warps, kStreamWarps, S::MINB), kStreamWarps * 32, rows, st>>>(c);
    return cudaGetLastError();
  });
}

// Warp w of n_warps takes items [part[w], part[w+1]), the shares balanced by
// cost: pre[x] is the summed cost of the items before x (over all minibatches).
__global__ void __launch_bounds__(256) stream_partition_kernel(const int64_t* __restrict__ pre, int32_t n_items,
                                                               int32_t n_warps, int32_t* __restrict__ part) {
  const int32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w > n_warps) return;
  int32_t lo = 0, hi = n_items;
  if (w == n_warps) {
    lo = n_items;
  } else {
    const int64_t target = pre[0] + (int64_t)((double)(pre[n_items] - pre[0]) * w / n_warps);
    while (lo < hi) {
      const int32_t m = lo + (hi - lo) / 2;
      if (pre[m] >= target) {
        hi = m;
      } else {
        lo = m + 1;
      }
    }
  }
  part[w] = lo;
}

cudaError_t launch_stream_partition(const int64_t* pre, int64_t n_items, int64_t n_warps, int32_t* part,
                                    cudaStream_t st) {
  stream_partition_kernel<<<(unsigned)(n_warps / 256 + 1), 256, 0, st>>>(pre, (int32_t)n_items, (int32_t)n_warps,
                                                                        part);
  return cudaGetLastError();
}

cudaError_t launch_row_refresh(const RowRefreshArgs& a, cudaStream_t st) {
  if (a.n_items <= 0) return cudaSuccess;
  row_refresh_kernel<<<grid_for(a.n_items, 32, 8), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_heavy_merge(const HeavyMergeArgs& a, cudaStream_t st) {
  if (a.n_heavy <= 0) return cudaSuccess;
  heavy_merge_kernel<<<grid_for(a.n_heavy, 8, 8), 256, 0, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_item_merge(const ItemMergeArgs& a, cudaStream_t st) {
  const int64_t work = std::max<int64_t>((int64_t)a.n_items * (a.K >> 2), a.do_schedule ? a.sched.P : 0);
  if (work <= 0) return cudaSuccess;
  // Every thread's loads are independent, so the whole merge is one set of
  // in-flight requests.  Eight (item, slice) pairs per thread: more loads in
  // flight per thread beat more threads with one each (0.019 against
  // 0.029 ms per clock on mid; 74 against 207 us on a 200k-item table).
  item_merge_kernel<8><<<(unsigned)std::min<int64_t>((work + 2047) / 2048, (int64_t)1 << 30), 256, 0, st>>>(a);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Objective (Sec. 3.1, Sec. 5) over all entries: sum e^2 and
// sum [e^2 + lambda(|L_i|^2 + |R_j|^2)], fp32 residuals, fp64 sums.
// One warp per entry.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) objective_kernel(const float* __restrict__ slot, int64_t n_users, int32_t K,
                                                        const int32_t* __restrict__ rec_u,
                                                        const int32_t* __restrict__ rec_j,
                                                        const float* __restrict__ rec_D, int64_t n_obs, float lambda,
                                                        double* out2) {
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int32_t K4 = K >> 2;
  const float4* t4 = reinterpret_cast<const float4*>(slot);
  double s1 = 0.0, s2 = 0.0;
  for (int64_t k = warp; k < n_obs; k += nwarps) {
    const float4* L = t4 + (int64_t)rec_u[k] * K4;
    const float4* R = t4 + (n_users + rec_j[k]) * K4;
    float dot = 0.f, nl = 0.f, nr = 0.f;
    for (int32_t q = lane; q < K4; q += 32) {
      const float4 l = L[q], r = R[q];
      dot += dot4(l, r);
      nl += dot4(l, l);
      nr += dot4(r, r);
    }
    dot = group_sum<32>(dot, 0xffffffffu);
    nl = group_sum<32>(nl, 0xffffffffu);
    nr = group_sum<32>(nr, 0xffffffffu);
    if (lane == 0) {
      const double e = (double)(rec_D[k] - dot);
      s1 += e * e;
      s2 += e * e + (double)lambda * ((double)nl + (double)nr);
    }
  }
  __shared__ double sh[2][8];
  const int w = threadIdx.x >> 5;
  if (lane == 0) {
    sh[0][w] = s1;
    sh[1][w] = s2;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    double x = 0.0, y = 0.0;
    for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
      x += sh[0][i];
      y += sh[1][i];
    }
    atomicAdd(out2, x);
    atomicAdd(out2 + 1, y);
  }
}

cudaError_t launch_objective(const float* slot, int64_t n_users, int32_t K, const int32_t* rec_u, const int32_t* rec_j,
                             const float* rec_D, int64_t n_obs, float lambda, double* out2, cudaStream_t st) {
  cudaError_t err = cudaMemsetAsync(out2, 0, 2 * sizeof(double), st);
  if (err != cudaSuccess || n_obs == 0) return err;
  objective_kernel<<<grid_for(n_obs, 8, 16), 256, 0, st>>>(slot, n_users, K, rec_u, rec_j, rec_D, n_obs, lambda, out2);
  return cudaGetLastError();
}

}  // namespace esspt
