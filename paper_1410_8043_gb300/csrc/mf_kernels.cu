// Matrix-factorisation SGD on the version ring (Sec. 3.1 updates under the
// SSP / ESSP read schedule).  One clock is:
//   sgd_stream_kernel   every user with entries (its row of version c,
//                       written once), every chunk of a very active one, and
//                       the rows of users without entries, carried from
//                       version c-1 to version c unless the ring already
//                       holds them;
//   clock_merge_kernel  the Clock() merge of the item rows and of the rows of
//                       the very active users.
// Item-row (and heavy-user) deltas are summed, unscaled, into zero-initialised
// replica rows so that popular rows spread their fp32 reductions over many
// L2 addresses; the merges apply eta, the hot-row scale and the sum of the
// replicas, then clear them for the next clock.
#include <algorithm>
#include <type_traits>

#include "chained.cuh"
#include "copy_idle.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "schedule.cuh"

namespace esspt {

namespace {

__device__ __forceinline__ float4 f4_zero() { return make_float4(0.f, 0.f, 0.f, 0.f); }

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

__device__ __forceinline__ void flush_loss(double* out, double x, int lane) {
  if (out == nullptr) return;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
  if (lane == 0 && x != 0.0) atomicAdd(out, x);
}

}  // namespace

constexpr int kStreamWarps = 4;   // warps per block
constexpr int kChunkSteps = 8;    // steps whose records are fetched together
constexpr int kMetaRounds = 8;    // rounds in the ring of item metadata

// One clock of MF-SGD over minibatch b.  The work list holds one item per user
// with 1..kHeavy entries and one per 64-entry chunk of a heavy user, sorted by
// length within tiles of consecutive users.  A warp walks one contiguous range
// of items in rounds of 32/G: each row group of G lanes (NV float4 slices of a
// row per lane, slice glane + t G on lane glane) takes one item, and the groups
// step through their items' entries together, E entries per group and step:
//   e = D - L.R,  gL += e R,  dR[dst] += e L - lambda R
// At the end of a round every group closes its item: a user's row of version c
// = base + eta s (gL - n lambda L), written once; a chunk's partial sum goes,
// unscaled, into its replica row of dL.  Which entries a step takes is known
// when the data are loaded, so the layout holds them in that order, those of a
// step side by side, and the stream runs on across rounds.
//
// The kernels that this one replaced took 80..92% of their time with the item
// rows served by L1 and the reductions left out: they waited on instruction
// issue and on the rows' latency.  So the groups of a warp share every
// instruction, on packed fp32 pairs (fma.rn.f32x2), with constant offsets from
// one pointer per row, and the item rows are gathered ahead:
//   rows of up to 64 values (E = 2): by cp.async, PF steps ahead (every lane
//     copies and reads its own slices only, so no barrier stands between); two
//     entries share a step's control and its shuffles;
//   wider rows (E = 1): in registers, one step ahead.  Their 256..2048 bytes
//     per entry through shared memory as well would make the SM's load/store
//     data path the limit (480k x 18k, K = 100: 480 us per clock against 440).
//     What bounds them is the SM's outgoing port, busy in 86% of the cycles that
//     L1 is active (K = 100): 12.5 of an entry's 21 cycles there are its reduction,
//     at 32 bytes per cycle, the rest row requests, entries and user rows.
template <int G, int NV, int E, int PF, int MINB, int HOT>
__global__ void __launch_bounds__(kStreamWarps * 32, MINB) sgd_stream_kernel(StreamArgs c) {
  constexpr int kGpw = 32 / G;
  constexpr int kPlaces = kGpw * E;          // entries per step of the warp
  constexpr int kRing = 2 * kChunkSteps;     // steps whose records are at hand
  static_assert(PF <= 3, "a chunk of records must have arrived when the gathers reach it");
  static_assert(E == 2 || (E == 1 && PF == 1 && HOT == 0), "one entry per step: rows in registers, one step ahead");
  __shared__ __align__(16) float4 stageL[kStreamWarps][NV][32];
  __shared__ __align__(16) float4 stageB[kStreamWarps][NV][32];
  __shared__ __align__(16) float4 rowsR[E == 2 ? kStreamWarps : 1][PF + 1][E][NV][E == 2 ? 32 : 1];
  __shared__ __align__(16) uint32_t recX[kStreamWarps][kRing * kPlaces];
  __shared__ __align__(16) uint32_t recYZ[kStreamWarps][kRing * kPlaces * 2];
  __shared__ __align__(16) int4 metas[kStreamWarps][kMetaRounds][kGpw];
  // per warp and lane: the summed updates of the minibatch's hot items
  __shared__ __align__(16) float4 hot[HOT > 0 ? kStreamWarps : 1][HOT > 0 ? HOT : 1][NV][HOT > 0 ? 32 : 1];
  const SgdArgs& a = c.a;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int glane = lane & (G - 1), grp = lane / G;
  const int32_t K4 = a.K >> 2;
  const bool last_on = glane + (NV - 1) * G < K4;  // the lane's last slice lies inside the row
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // Sum of e^2: of the round, and of the rounds before with the rounding error
  // kept beside it (two-sum, Knuth, TAOCP vol. 2, 4.2.2): a lane adds thousands
  // of squares, and one fp32 sum of them was off by 6.5e-7 on 10M x 1M, K = 64.
  float loss = 0.f, loss_sum = 0.f, loss_lost = 0.f;
  auto fold_loss = [&]() {
    const float t = loss_sum + loss, b = t - loss_sum;
    loss_lost += (loss_sum - (t - b)) + (loss - b);
    loss_sum = t;
    loss = 0.f;
  };
  await_previous_kernel();

  // Half of the warps copy idle rows first, the others last: the copy's DRAM
  // traffic runs beside the other warps' arithmetic.
  if (warp & 1) copy_idle_users<G, NV>(a, warp, nwarps, lane);

  int32_t xr = 0, xb = 0;
  uint32_t s0 = 0, s1 = 0;
  if (warp < c.n_warps) {
    const int4 p0 = __ldg(c.part + warp);
    xr = p0.x;
    xb = p0.y;
    s0 = (uint32_t)p0.z;
    s1 = (uint32_t)p0.w;
  }
  if (s0 < s1) {
    const int64_t slot4 = a.n_rows * K4;
    float4* ring4 = reinterpret_cast<float4*>(a.ring) + glane;
    float4* dRq = reinterpret_cast<float4*>(a.dR) + glane;
    const uint64_t pol = policy_evict_first();
    const u64 nlam = pack2(-a.lambda, -a.lambda);

    auto load_item = [&](int32_t r0) {  // the group's item of the round that starts at item r0
      const int32_t x = r0 + grp;
      return x < xb ? __ldg(c.items + x) : make_int4(0, 0, -2, 0);
    };
    // Item as kept for its round: x = user, y = steps of the round, z as in
    // the list, w = its read version's ring slot and its length.
    auto put_meta = [&](int at, const int4& it) {
      const int32_t n = it.w >> 16;
      const int32_t steps = __reduce_max_sync(0xffffffffu, (n + E - 1) / E);
      const int32_t vs = a.row_mode ? a.user_slot[it.x] : a.vslot[it.w & 0xffff];
      if (glane == 0) metas[wib][at][grp] = make_int4(it.x, steps, it.z, vs << 7 | n);
    };
    auto item_rows = [&](int32_t vs) -> const float4* {
      return a.row_mode ? ring4 : ring4 + vs * slot4 + (int64_t)a.n_users * K4;
    };
    // Copy user u's row of ring slot vs.
    auto stage = [&](float4(&to)[NV][32], int32_t vs, int32_t u, bool on) {
      const float4* row = ring4 + vs * slot4 + (int64_t)u * K4;
#pragma unroll
      for (int k = 0; k < NV; ++k) cp_async16_hint_if(&to[k][lane], row + k * G, on && (k < NV - 1 || last_on), pol);
    };
    // The records of kChunkSteps steps from step s (s - s0 a multiple of it).
    auto fetch_records = [&](uint32_t s) {
      const int half = (s - s0) & kChunkSteps;
#pragma unroll
      for (int l0 = 0; l0 < kChunkSteps * kPlaces; l0 += 128) {
        const int l = l0 + 4 * lane;
        const bool on = l < kChunkSteps * kPlaces && s + l / kPlaces < s1;
        cp_async16_hint_if(&recX[wib][half * kPlaces + l], c.x + (int64_t)s * kPlaces + l, on, pol);
      }
#pragma unroll
      for (int l0 = 0; l0 < kChunkSteps * kPlaces * 2; l0 += 128) {
        const int l = l0 + 4 * lane;
        const bool on = l < kChunkSteps * kPlaces * 2 && s + l / (2 * kPlaces) < s1;
        cp_async16_hint_if(&recYZ[wib][half * kPlaces * 2 + l], c.yz + (int64_t)s * kPlaces * 2 + l, on, pol);
      }
    };

#pragma unroll
    for (int k = 0; k < NV; ++k) {  // slices past the row end stay zero
      stageL[wib][k][lane] = f4_zero();
      if constexpr (E == 2)
#pragma unroll
        for (int q = 0; q <= PF; ++q) rowsR[wib][q][0][k][lane] = rowsR[wib][q][1][k][lane] = f4_zero();
#pragma unroll
      for (int h = 0; h < HOT; ++h) hot[wib][h][k][lane] = f4_zero();
    }
    fetch_records(s0);
    fetch_records(s0 + kChunkSteps);
    constexpr int kAhead = PF + 2;  // rounds whose metadata are at hand
    static_assert(kAhead < kMetaRounds, "the ring of metadata");
#pragma unroll
    for (int d = 0; d < kAhead; ++d) put_meta(d, load_item(xr + d * kGpw));
    int4 far = load_item(xr + kAhead * kGpw);
    cp_async_wait_all();
    __syncwarp();

    // The gathers' place: round in the ring of metadata, steps left of it, its item rows.
    int frnd = 0, fleft = metas[wib][0][grp].y;
    const float4* fR = item_rows(metas[wib][0][grp].w >> 7);
    auto f_next = [&]() {
      if (--fleft == 0) {
        frnd = (frnd + 1) & (kMetaRounds - 1);
        const int4 m = metas[wib][frnd][grp];
        fleft = m.y;
        fR = item_rows(m.w >> 7);
      }
    };

    // Current round.
    f2x2 L[NV], gL[NV];
    int32_t cur_u = 0, cur_z = 0, cur_n = 0, cur_vs = 0, left = 0;
    int rnd = 0;
    bool quick = false;  // a round of so few steps that its staged rows may not be there at its end
    auto open_round = [&]() {
      const int4 m = metas[wib][rnd][grp];
      cur_u = m.x;
      left = m.y;
      cur_z = m.z;
      cur_n = m.w & 127;
      cur_vs = m.w >> 7;
      quick = left <= PF;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        L[k] = lds_f2x2(&stageL[wib][k][lane]);
        gL[k] = f2x2{0ull, 0ull};
      }
      const int4 m1 = metas[wib][(rnd + 1) & (kMetaRounds - 1)][grp];
      stage(stageL[wib], m1.w >> 7, m1.x, xr + kGpw < xb && (m1.w & 127) > 0);
      stage(stageB[wib], a.slot_base, cur_u, cur_z == -1 && cur_vs != a.slot_base);
      put_meta((rnd + kAhead) & (kMetaRounds - 1), far);
      far = load_item(xr + (kAhead + 1) * kGpw);
      __syncwarp();
    };
    auto close_round = [&]() {
      if (E == 1 || quick) cp_async_wait_all();
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
          if (!same) b = lds_f2x2(&stageB[wib][k][lane]);
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
    // True once the warp's stream is done.
    auto step_done = [&]() -> bool {
      if (--left > 0) return false;
      close_round();
      fold_loss();
      xr += kGpw;
      if (xr >= xb) return true;
      rnd = (rnd + 1) & (kMetaRounds - 1);
      open_round();
      return false;
    };
    auto dot_part = [&](const f2x2(&R)[NV]) -> float {
      u64 p = mul2(L[0].lo, R[0].lo);
      p = fma2(L[0].hi, R[0].hi, p);
#pragma unroll
      for (int k = 1; k < NV; ++k) {
        p = fma2(L[k].lo, R[k].lo, p);
        p = fma2(L[k].hi, R[k].hi, p);
      }
      return sum2(p);
    };
    // gL and the item update of an entry with residual e, y its record's word.
    auto update = [&](float e, uint32_t y, const f2x2(&R)[NV]) {
      const u64 ee = pack2(e, e);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        gL[k].lo = fma2(ee, R[k].lo, gL[k].lo);
        gL[k].hi = fma2(ee, R[k].hi, gL[k].hi);
      }
      if (HOT > 0 && (y & 1u)) {
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          float4* h = &hot[wib][y >> 1][k][lane];
          const f2x2 v = lds_f2x2(h);
          st_f2x2(h, add2(v.lo, fma2(ee, L[k].lo, mul2(nlam, R[k].lo))),
                   add2(v.hi, fma2(ee, L[k].hi, mul2(nlam, R[k].hi))));
        }
      } else {
        float4* out = dRq + y;
#pragma unroll
        for (int k = 0; k < NV; ++k)
          red_add_f2x2_if(out + k * G, fma2(ee, L[k].lo, mul2(nlam, R[k].lo)),
                          fma2(ee, L[k].hi, mul2(nlam, R[k].hi)), k < NV - 1 || last_on);
      }
    };

    {
      const int4 m = metas[wib][0][grp];
      stage(stageL[wib], m.w >> 7, m.x, (m.w & 127) > 0);
    }
    if constexpr (E == 2) {
      // Gather the item rows of step t into place q of the ring of rows.
      auto gather = [&](uint32_t t, int q) {
        if (t < s1) {
          const uint2 x = *reinterpret_cast<const uint2*>(&recX[wib][(((t - s0) & (kRing - 1)) * kGpw + grp) * 2]);
#pragma unroll
          for (int k = 0; k < NV; ++k) {
            cp_async16_if(&rowsR[wib][q][0][k][lane], fR + x.x + k * G, x.x != kNoRecord && (k < NV - 1 || last_on));
            cp_async16_if(&rowsR[wib][q][1][k][lane], fR + x.y + k * G, x.y != kNoRecord && (k < NV - 1 || last_on));
          }
          f_next();
        }
      };
#pragma unroll
      for (int q = 0; q < PF; ++q) gather(s0 + q, q);
      cp_async_wait_all();
      open_round();
      int q = 0;  // place of step s in the ring of rows
      const bool hi = lane & (G / 2);  // this lane ends up with the second entry's dot product
      for (uint32_t s = s0;; ++s) {
        gather(s + PF, q == 0 ? PF : q - 1);
        if (((s - s0) & (kChunkSteps - 1)) == 0 && s > s0) fetch_records(s + kChunkSteps);
        cp_async_commit();
        cp_async_wait<PF>();
        __syncwarp();
        const uint4 r = *reinterpret_cast<const uint4*>(&recYZ[wib][(((s - s0) & (kRing - 1)) * kGpw + grp) * 4]);
        f2x2 R0[NV], R1[NV];
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          R0[k] = lds_f2x2(&rowsR[wib][q][0][k][lane]);
          R1[k] = lds_f2x2(&rowsR[wib][q][1][k][lane]);
        }
        q = q == PF ? 0 : q + 1;
        const float p0 = dot_part(R0), p1 = dot_part(R1);
        float dot = hi ? p1 : p0;
        dot += __shfl_xor_sync(0xffffffffu, hi ? p0 : p1, G / 2);
#pragma unroll
        for (int off = G / 4; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        const float e = __uint_as_float(hi ? r.w : r.z) - dot;
        const float o = __shfl_xor_sync(0xffffffffu, e, G / 2);
        if (r.x != kNoRecord) update(hi ? o : e, r.x, R0);
        if (r.y != kNoRecord) update(hi ? e : o, r.y, R1);
        if ((hi ? r.y : r.x) != kNoRecord) loss += e * e;
        if (step_done()) break;
      }
      if (glane % (G / 2) != 0) loss_sum = loss_lost = 0.f;
    } else {
      f2x2 Ra[NV], Rb[NV];
#pragma unroll
      for (int k = 0; k < NV; ++k) Ra[k] = Rb[k] = f2x2{0ull, 0ull};
      auto gather = [&](uint32_t t, f2x2(&R)[NV]) {
        if (t < s1) {
          const uint32_t x = recX[wib][((t - s0) & (kRing - 1)) * kGpw + grp];
#pragma unroll
          for (int k = 0; k < NV; ++k) ld_f2x2_if(R[k], fR + x + k * G, x != kNoRecord && (k < NV - 1 || last_on));
          f_next();
        }
      };
      gather(s0, Ra);
      cp_async_wait_all();
      open_round();
      auto step = [&](uint32_t s, const f2x2(&Rc)[NV], f2x2(&Rn)[NV]) -> bool {
        if (((s - s0) & (kChunkSteps - 1)) == kChunkSteps - 1) {  // the next step's records, fetched 8 steps ago
          cp_async_wait_all();
          __syncwarp();
        }
        gather(s + 1, Rn);
        if (((s - s0) & (kChunkSteps - 1)) == 0 && s > s0) fetch_records(s + kChunkSteps);
        const uint2 r = *reinterpret_cast<const uint2*>(&recYZ[wib][(((s - s0) & (kRing - 1)) * kGpw + grp) * 2]);
        float dot = dot_part(Rc);
#pragma unroll
        for (int off = G / 2; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
        if (r.x != kNoRecord) {
          const float e = __uint_as_float(r.y) - dot;
          loss += e * e;
          update(e, r.x, Rc);
        }
        return step_done();
      };
      for (uint32_t s = s0;; s += 2) {
        if (step(s, Ra, Rb)) break;
        if (step(s + 1, Rb, Ra)) break;
      }
      if (glane != 0) loss_sum = loss_lost = 0.f;
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
  // (an infinite or NaN sum has no rounding error)
  flush_loss(a.sq_loss, isfinite(loss_sum) ? (double)loss_sum + (double)loss_lost : (double)loss_sum, lane);
}

// The Clock() merge (Sec. 2.1 additive updates, Sec. 4 server clock):
//   R^c_j = R^base_j + eta s_j (sum of j's replica rows of dR)
// and, for the heavy users, L^c_i likewise from dL; replicas are cleared for
// the next clock.  Warps take three kinds of task, the long ones first:
//   an item with extra replicas or a heavy user: the row groups of the warp
//     split its replica rows, each with all its loads of a pass in flight;
//   kUnit other items: base row and replica row of each, read and written once;
//     an item without entries is only copied forward, and not even that when
//     the ring already holds it (as for idle users).
// With do_schedule the first P threads also compute the next clock's read
// versions (the SGD kernel of this clock, the only reader of v, has finished).
// DRAM bounds the third kind: 1M items of 64 values move 1.0 GB.  One thread
// per slice with the extra replicas in line, eight slices in flight at one
// block per SM, took 353 us there and a launch for the heavy users 50 more.
template <int G, int NV>
__global__ void __launch_bounds__(256, 3) clock_merge_kernel(MergeArgs a) {
  constexpr int kGpw = 32 / G;
  constexpr int kBatch = NV >= 3 ? 1 : 4 / NV;  // items per group in flight
  constexpr int kUnit = kGpw * kBatch;          // items per task, <= 32
  constexpr int kRows = kBatch;                 // replica rows per group in flight
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  await_previous_kernel();
  if (a.do_schedule)
    for (int64_t p = tid; p < a.sched.P; p += nth) schedule_worker(a.sched, (int32_t)p);
  const int lane = threadIdx.x & 31, glane = lane & (G - 1), grp = lane / G;
  const int32_t K4 = a.K >> 2;
  const bool last_on = glane + (NV - 1) * G < K4;
  float4* ring4 = reinterpret_cast<float4*>(a.ring) + glane;
  const float4* base4 = ring4 + (int64_t)a.slot_base * a.n_rows * K4;
  float4* out4 = ring4 + (int64_t)a.slot_out * a.n_rows * K4;
  const int64_t nwarps = nth >> 5, lists = a.n_popular + a.n_heavy;
  int64_t task = tid >> 5;

  for (; task < lists; task += nwarps) {
    const bool item = task < a.n_popular;
    const int4 d = __ldg(item ? a.popular + task : a.heavy + (task - a.n_popular));
    float4* rows = reinterpret_cast<float4*>(item ? a.dR : a.dL) + glane;
    const int64_t ld = item ? a.dR_ld : K4, row = item ? (int64_t)a.n_users + d.x : (int64_t)d.x;
    const int32_t n = item ? __ldg(a.item_cnt + d.x) : d.w;
    float4 acc[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) acc[k] = f4_zero();
    for (int32_t r0 = grp; r0 < d.z; r0 += kRows * kGpw) {
      float4 x[kRows][NV];
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int32_t r = r0 + u * kGpw;
        const float4* p = rows + (r == 0 ? (int64_t)d.x : (int64_t)d.y + r - 1) * ld;
#pragma unroll
        for (int k = 0; k < NV; ++k) x[u][k] = r < d.z && (k < NV - 1 || last_on) ? p[k * G] : f4_zero();
      }
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        const int32_t r = r0 + u * kGpw;
        float4* p = rows + (r == 0 ? (int64_t)d.x : (int64_t)d.y + r - 1) * ld;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          acc[k] = f4_add(acc[k], x[u][k]);
          if (r < d.z && (k < NV - 1 || last_on)) p[k * G] = f4_zero();
        }
      }
    }
    const float sc = a.eta * cap_scale(a.cap, n);
#pragma unroll
    for (int k = 0; k < NV; ++k) {
#pragma unroll
      for (int off = G; off < 32; off <<= 1) {
        acc[k].x += __shfl_xor_sync(0xffffffffu, acc[k].x, off);
        acc[k].y += __shfl_xor_sync(0xffffffffu, acc[k].y, off);
        acc[k].z += __shfl_xor_sync(0xffffffffu, acc[k].z, off);
        acc[k].w += __shfl_xor_sync(0xffffffffu, acc[k].w, off);
      }
      if (grp == 0 && (k < NV - 1 || last_on)) out4[row * K4 + k * G] = f4_axpy(sc, acc[k], base4[row * K4 + k * G]);
    }
    if (lane == 0 && n > 0) (item ? a.chg_item : a.chg)[d.x] = a.clock;
  }

  float4* dR4 = reinterpret_cast<float4*>(a.dR) + glane;
  const bool may_skip = a.clock > a.copy_all_until;
  const int64_t units = ((int64_t)a.n_items + kUnit - 1) / kUnit;
  // What to do with this lane's item of a unit: nothing (it has extra replicas,
  // or the ring holds its row), copy it (-1: no entries), or merge n entries.
  auto look = [&](int64_t unit) -> int32_t {
    const int64_t j = unit * kUnit + lane;
    if (lane >= kUnit || j >= a.n_items || __ldg(a.item_rep + j + 1) > __ldg(a.item_rep + j)) return 0;
    const int32_t n = __ldg(a.item_cnt + j);
    if (n > 0) return n;
    return may_skip && a.clock - a.chg_item[j] >= a.nslots ? 0 : -1;
  };
  int64_t unit = task - lists;
  int32_t todo = unit < units ? look(unit) : 0;
  for (; unit < units; unit += nwarps) {
    const int32_t now = todo;
    todo = unit + nwarps < units ? look(unit + nwarps) : 0;
    if (now > 0) a.chg_item[unit * kUnit + lane] = a.clock;
    float4 x[kBatch][NV], b[kBatch][NV];
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int32_t n = __shfl_sync(0xffffffffu, now, u * kGpw + grp);
      const int64_t j = unit * kUnit + u * kGpw + grp;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const bool in = k < NV - 1 || last_on;
        x[u][k] = n > 0 && in ? dR4[j * a.dR_ld + k * G] : f4_zero();
        b[u][k] = n != 0 && in ? base4[(a.n_users + j) * K4 + k * G] : f4_zero();
      }
    }
#pragma unroll
    for (int u = 0; u < kBatch; ++u) {
      const int32_t n = __shfl_sync(0xffffffffu, now, u * kGpw + grp);
      const int64_t j = unit * kUnit + u * kGpw + grp;
      const float sc = a.eta * cap_scale(a.cap, n);
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const bool in = k < NV - 1 || last_on;
        if (n > 0 && in) dR4[j * a.dR_ld + k * G] = f4_zero();
        if (n != 0 && in) out4[(a.n_users + j) * K4 + k * G] = f4_axpy(sc, x[u][k], b[u][k]);
      }
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

}  // namespace

int grid_for(int64_t work_items, int64_t per_block, int max_per_sm) {
  const int64_t want = (work_items + per_block - 1) / per_block;
  return (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sm_count() * max_per_sm));
}

namespace {

// Row-group shape for K: G lanes per row (a power of two) and NV float4 slices
// per lane, G (NV - 1) < K/4 <= G NV; E entries per step and PF steps of gathers
// ahead (see the kernel); the blocks per SM it is compiled for.  Eight lanes
// read 128 consecutive bytes per load, a whole line; wider groups only where
// NV = 4 slices per lane do not hold the row.  Measured (us per clock):
//   K = 32, 200k x 30k: PF 2 with 6 blocks 68..75 over three inputs, with 7 (it
//     spills) 74..78, PF 1 with 7 blocks 74..77; one entry per step more; K = 28,
//     1M x 100k: 197, 195, 195;
//   K = 48, 300k x 40k: PF 1 with 5 blocks 107, PF 2 with 4 blocks 114; one
//     entry per step 108..118; 10M x 1M, K = 64: 2630, 2650; 2720..2810;
//   K = 100, 480k x 18k: 4 blocks 441..450, 3 blocks 470, 5 blocks spill (785).
template <int G_, int NV_, int E_, int PF_, int MINB_, int HOT_ = 0>
struct StreamShape {
  static constexpr int G = G_, NV = NV_, E = E_, PF = PF_, MINB = MINB_, HOT = HOT_, GPW = 32 / G_;
};
template <typename F>
auto dispatch_stream(int32_t K, F&& f) {
  const int32_t K4 = K / 4;
  if (K4 <= 4) return f(StreamShape<4, 1, 2, 2, 6>{});
  if (K4 <= 8) return f(StreamShape<8, 1, 2, 2, 6>{});
  if (K4 <= 16) return f(StreamShape<8, 2, 2, 1, 5, kHot>{});
  if (K4 <= 24) return f(StreamShape<8, 3, 1, 1, 5>{});
  if (K4 <= 32) return f(StreamShape<8, 4, 1, 1, 4>{});
  if (K4 <= 48) return f(StreamShape<16, 3, 1, 1, 5>{});
  if (K4 <= 64) return f(StreamShape<16, 4, 1, 1, 4>{});
  if (K4 <= 96) return f(StreamShape<32, 3, 1, 1, 5>{});
  return f(StreamShape<32, 4, 1, 1, 4>{});
}

// Blocks of the stream kernel: warps for the work list, and one per 32 users
// for the forward copy, up to one resident wave.
template <typename S>
int stream_blocks(int64_t n_warps, int64_t n_users) {
  return grid_for(std::max<int64_t>(n_warps, (n_users + 31) / 32), kStreamWarps, S::MINB);
}

}  // namespace

bool stream_is_small(int32_t K, int64_t n_warps, int64_t n_users) {
  return dispatch_stream(K, [&](auto s) { return stream_blocks<decltype(s)>(n_warps, n_users) <= sm_count(); });
}

int64_t stream_max_warps(int32_t K) {
  return dispatch_stream(K, [](auto s) { return (int64_t)sm_count() * s.MINB * kStreamWarps; });
}

StreamGeometry stream_geometry(int32_t K) {
  return dispatch_stream(K, [](auto s) { return StreamGeometry{s.GPW, s.E}; });
}

cudaError_t launch_sgd_stream(const StreamArgs& c, cudaStream_t st) {
  return dispatch_stream(c.a.K, [&](auto s) {
    using S = decltype(s);
    const auto kernel = sgd_stream_kernel<S::G, S::NV, S::E, S::PF, S::MINB, S::HOT>;
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
    // The SGD kernel starts while the kernel before it, in a run of clocks the
    // merge, drains; the merge only on clocks of at most one block per SM.
    // 2k x 1k, K = 16: 14.0 us per clock with neither, 10.6 with the first, 8.7
    // with both.  Larger clocks lose with both (480k x 18k, K = 100: 445 us, 520
    // with both; 10M x 1M, K = 64: 2480, 2700).
    return launch_chained(kernel, stream_blocks<S>(c.n_warps, c.a.n_users), kStreamWarps * 32, st, true, c);
  });
}

cudaError_t launch_clock_merge(const MergeArgs& a, cudaStream_t st) {
  return dispatch_stream(a.K, [&](auto s) {
    using S = decltype(s);
    const int64_t unit = S::GPW * (S::NV >= 3 ? 1 : 4 / S::NV);
    const int64_t warps = a.n_popular + a.n_heavy + (a.n_items + unit - 1) / unit;
    const int64_t most = std::max<int64_t>(warps, a.do_schedule ? (a.sched.P + 31) / 32 : 0);
    return launch_chained(clock_merge_kernel<S::G, S::NV>, grid_for(most, 8, 3), 256, st, a.chained != 0, a);
  });
}

}  // namespace esspt
