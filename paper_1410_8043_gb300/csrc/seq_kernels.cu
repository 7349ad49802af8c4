// Sequential (read-my-writes) MF-SGD of one clock: each worker walks its own
// entries in order and reads L_i and R_j from its read version plus its own
// updates of this clock so far, as the per-entry SGD of Sec. 3.1 runs inside
// a worker (Sec. 5); the workers' summed changes then join the Clock() merge.
// An entry depends on the worker's earlier entries of the same user and of the
// same item.  One warp per worker takes them all in turn, though entries that
// share neither could go side by side (64k entries, K = 64, 16 workers: about
// 4000 entries per worker, 230..330 of them in the longest chain of dependent
// ones): this is a semantic variant, not the data-parallel hot path.
#include <algorithm>
#include <type_traits>

#include "copy_idle.cuh"
#include "internal.h"
#include "ptx.cuh"

namespace esspt {

namespace {

constexpr int kSegment = 128;  // entries queued at a time

__device__ __forceinline__ float seq_cap_scale(int32_t cap, int32_t n) {
  return (cap > 0 && n > cap) ? (float)cap / (float)n : 1.f;
}

__device__ __forceinline__ f2x2 load_row(const float4* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return f2x2{v.x, v.y};
}

// A queued entry: x = user, y = item, z = value, w = kFirst / kLast entry of its
// user, kRepeat where one of the next three has the same item.
constexpr int kFirst = 1, kLast = 2, kRepeat = 4;

// Blocks [0, P): worker p's chain, walked by warp 0, its queue filled by warp 1.
// Blocks from P on copy the idle users' rows.
//
// The length of the walk bounds it, so an entry holds as little as it can: the dot
// product and two fused updates.  The rows of the read version (item's, user's
// at its first entry, and the base row at its last) come by cp.async AHEAD
// entries early, the worker's change to the item's row in registers three
// early; where one of those three has the same item, the entry's result
// replaces what was loaded (no other worker writes it).  The second warp turns
// the worker's users into a queue of entries one segment ahead.  64k entries,
// K = 64, 16 workers: 2.9 ms with every load in the chain, 2.0 with rows two
// entries early.
template <int G, int NV>
__global__ void __launch_bounds__(64) seq_users_kernel(SeqArgs s) {
  constexpr int kRing = NV * G <= 64 ? 8 : 4, AHEAD = kRing - 1;
  const SgdArgs& a = s.a;
  const int lane = threadIdx.x & 31;
  if (blockIdx.x >= s.P) {
    const int64_t first = (int64_t)(blockIdx.x - s.P) * 2 + (threadIdx.x >> 5);
    copy_idle_users<G, NV>(a, first, (int64_t)(gridDim.x - s.P) * 2, lane);
    return;
  }
  __shared__ __align__(16) float4 ring[kRing][3][NV][G];  // rows of the read version: item's, user's; base row
  __shared__ int4 queue[2][kSegment];
  __shared__ int32_t queued[2];
  const int32_t p = blockIdx.x;
  const int glane = lane & (G - 1);
  const int32_t K4 = a.K >> 2;
  const bool mine_lane = lane < G;  // the other lanes only take part in the shuffles
  const bool last_on = mine_lane && glane + (NV - 1) * G < K4;
  const int64_t slot4 = a.n_rows * K4;
  float4* ring4 = reinterpret_cast<float4*>(a.ring) + glane;
  const float4* X = ring4 + (int64_t)(__ldg(s.v + p) % a.nslots) * slot4;
  const float4* XR = X + (int64_t)a.n_users * K4;
  const float4* base = ring4 + (int64_t)a.slot_base * slot4;
  float4* out = ring4 + (int64_t)a.slot_out * slot4;
  float4* mine = reinterpret_cast<float4*>(s.mine) + (int64_t)p * s.n_items * K4 + glane;
  const bool walker = threadIdx.x < 32;
  int32_t at = __ldg(s.wbase + p);             // filler: next user of the worker,
  const int32_t end = __ldg(s.wbase + p + 1);
  int32_t done = 0;                            // and its entries already queued
  float loss = 0.f;
  f2x2 L[NV], dL[NV];
  int32_t n = 0;
#pragma unroll
  for (int k = 0; k < NV; ++k) L[k] = dL[k] = f2x2{0ull, 0ull};

  auto fill = [&](int buf) {
    int32_t have = 0;
    while (have < kSegment && at < end) {
      const bool in = at + lane < end;
      const int32_t u = in ? __ldg(s.wuser + at + lane) : 0;
      int32_t beg = in ? __ldg(a.uoff + u) : 0;
      const int32_t stop = in ? __ldg(a.uoff + u + 1) : 0;
      const int32_t first = beg;
      if (lane == 0) beg += done;
      int32_t incl = stop - beg;  // entries of lanes 0 .. lane
#pragma unroll
      for (int off = 1; off < 32; off <<= 1) {
        const int32_t o = __shfl_up_sync(0xffffffffu, incl, off);
        if (lane >= off) incl += o;
      }
      const int32_t excl = incl - (stop - beg);
      const int32_t take = min(kSegment - have, __shfl_sync(0xffffffffu, incl, 31));
      for (int32_t t0 = 0; t0 < take; t0 += 32) {
        const int32_t t = t0 + lane;
        int own = 0;  // first lane with incl > t
#pragma unroll
        for (int h = 16; h > 0; h >>= 1)
          if (__shfl_sync(0xffffffffu, incl, min(own + h - 1, 31)) <= t) own += h;
        own = min(own, 31);
        const int32_t e = __shfl_sync(0xffffffffu, beg, own) + t - __shfl_sync(0xffffffffu, excl, own);
        const int32_t ou = __shfl_sync(0xffffffffu, u, own), of = __shfl_sync(0xffffffffu, first, own);
        const int32_t os = __shfl_sync(0xffffffffu, stop, own);
        if (t < take)
          queue[buf][have + t] = make_int4(ou, __ldg(s.rec_j + e), __float_as_int(__ldg(s.rec_D + e)),
                                           (e == of ? kFirst : 0) | (e + 1 == os ? kLast : 0));
      }
      have += take;
      // users wholly queued (users without entries too), and what is left of the next
      const int whole = __popc(__ballot_sync(0xffffffffu, in && incl <= take));
      const int32_t before = whole > 0 ? __shfl_sync(0xffffffffu, incl, whole - 1) : 0;
      done = take - before + (whole == 0 ? done : 0);
      at += whole;
    }
    __syncwarp();
    for (int32_t t = lane; t < have; t += 32) {
      const int32_t j = queue[buf][t].y;
      bool repeat = false;
      for (int32_t d = 1; d <= 3 && t + d < have; ++d) repeat |= queue[buf][t + d].y == j;
      if (repeat) queue[buf][t].w |= kRepeat;
    }
    if (lane == 0) queued[buf] = have;
  };
  const u64 pol = policy_evict_first();
  // Read-version rows of entry t of a segment, into its place of the ring.
  auto issue = [&](int buf, int32_t t, int32_t cnt) {
    if (t < cnt) {
      const int4 q = queue[buf][t];
      float4(*to)[NV][G] = ring[t & (kRing - 1)];
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        const bool on = k < NV - 1 ? mine_lane : last_on;
        cp_async16_if(&to[0][k][glane], XR + (int64_t)q.y * K4 + k * G, on);
        cp_async16_hint_if(&to[1][k][glane], X + (int64_t)q.x * K4 + k * G, on && (q.w & kFirst), pol);
        cp_async16_hint_if(&to[2][k][glane], base + (int64_t)q.x * K4 + k * G, on && (q.w & kLast), pol);
      }
    }
    cp_async_commit();
  };
  // The worker's change to the item row of entry t.
  auto load_mine = [&](f2x2(&M)[NV], int buf, int32_t t, int32_t cnt) {
    if (t >= cnt) return;
    const float4* m = mine + (int64_t)queue[buf][t].y * K4;
#pragma unroll
    for (int k = 0; k < NV; ++k)
      if (k < NV - 1 ? mine_lane : last_on) M[k] = load_row(m + k * G);
  };
  const u64 eta2 = pack2(a.eta, a.eta), nlam2 = pack2(-a.lambda, -a.lambda);
  // Entry t of a segment, M its item's change; M1 .. M3 those of the next three.
  auto walk = [&](f2x2(&M)[NV], f2x2(&M1)[NV], f2x2(&M2)[NV], f2x2(&M3)[NV], int buf, int32_t t, int32_t cnt) {
    load_mine(M3, buf, t + 3, cnt);
    issue(buf, t + AHEAD, cnt);
    cp_async_wait<AHEAD>();
    const int4 q = queue[buf][t];
    const float4(*row)[NV][G] = ring[t & (kRing - 1)];
    if (q.w & kFirst) {
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        L[k] = lds_f2x2(&row[1][k][glane]);
        dL[k] = f2x2{0ull, 0ull};
      }
      n = 0;
    }
    f2x2 R[NV];
    u64 acc = 0ull;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      const f2x2 x = lds_f2x2(&row[0][k][glane]);
      R[k] = f2x2{add2(x.lo, M[k].lo), add2(x.hi, M[k].hi)};
      acc = fma2(L[k].lo, R[k].lo, acc);
      acc = fma2(L[k].hi, R[k].hi, acc);
    }
    float dot = sum2(acc);
#pragma unroll
    for (int off = G / 2; off > 0; off >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, off);
    const float res = __int_as_float(q.z) - dot;
    loss += res * res;
    const u64 e2 = pack2(res, res);
    float4* m = mine + (int64_t)q.y * K4;
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      // eta (e R - lambda L) and eta (e L - lambda R)
      const u64 gll = mul2(eta2, fma2(e2, R[k].lo, mul2(nlam2, L[k].lo)));
      const u64 glh = mul2(eta2, fma2(e2, R[k].hi, mul2(nlam2, L[k].hi)));
      const u64 grl = mul2(eta2, fma2(e2, L[k].lo, mul2(nlam2, R[k].lo)));
      const u64 grh = mul2(eta2, fma2(e2, L[k].hi, mul2(nlam2, R[k].hi)));
      L[k] = f2x2{add2(L[k].lo, gll), add2(L[k].hi, glh)};
      dL[k] = f2x2{add2(dL[k].lo, gll), add2(dL[k].hi, glh)};
      M[k] = f2x2{add2(M[k].lo, grl), add2(M[k].hi, grh)};
      if (k < NV - 1 ? mine_lane : last_on) st_f2x2(m + k * G, M[k].lo, M[k].hi);
    }
    if (q.w & kRepeat) {
      const bool r1 = t + 1 < cnt && queue[buf][t + 1].y == q.y, r2 = t + 2 < cnt && queue[buf][t + 2].y == q.y,
                 r3 = t + 3 < cnt && queue[buf][t + 3].y == q.y;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        if (r1) M1[k] = M[k];
        if (r2) M2[k] = M[k];
        if (r3) M3[k] = M[k];
      }
    }
    ++n;
    if (q.w & kLast) {  // L_i^c = L_i^base + scale * (the user's summed change)
      const float sc = seq_cap_scale(a.cap, n);
      const u64 sc2 = pack2(sc, sc);
      float4* o = out + (int64_t)q.x * K4;
#pragma unroll
      for (int k = 0; k < NV; ++k)
        if (k < NV - 1 ? mine_lane : last_on) {
          const f2x2 b = lds_f2x2(&row[2][k][glane]);
          st_f2x2(o + k * G, fma2(sc2, dL[k].lo, b.lo), fma2(sc2, dL[k].hi, b.hi));
        }
      if (lane == 0) a.chg[q.x] = a.clock;
    }
  };

  f2x2 M0[NV], M1[NV], M2[NV], M3[NV];
#pragma unroll
  for (int k = 0; k < NV; ++k) M0[k] = M1[k] = M2[k] = M3[k] = f2x2{0ull, 0ull};
  for (int k = threadIdx.x; k < kRing * 3 * NV * G; k += 64) (&ring[0][0][0][0])[k] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (!walker) fill(0);
  __syncthreads();
  for (int buf = 0; queued[buf] > 0; buf ^= 1) {
    const int32_t cnt = queued[buf];
    if (walker) {
      // A segment starts with no change in flight: those it reads are stored.
      for (int32_t t = 0; t < AHEAD; ++t) issue(buf, t, cnt);
      load_mine(M0, buf, 0, cnt);
      load_mine(M1, buf, 1, cnt);
      load_mine(M2, buf, 2, cnt);
      for (int32_t t = 0; t < cnt; t += 4) {
        walk(M0, M1, M2, M3, buf, t, cnt);
        if (t + 1 < cnt) walk(M1, M2, M3, M0, buf, t + 1, cnt);
        if (t + 2 < cnt) walk(M2, M3, M0, M1, buf, t + 2, cnt);
        if (t + 3 < cnt) walk(M3, M0, M1, M2, buf, t + 3, cnt);
      }
      cp_async_wait_all();
    } else {
      fill(buf ^ 1);
    }
    __syncthreads();
  }
  if (a.sq_loss != nullptr && walker && lane == 0 && loss != 0.f) atomicAdd(a.sq_loss, (double)loss);
}

// Clock() merge of the item rows: R_j^c = R_j^base + scale_j * sum over
// workers (in worker order) of their changes to R_j.  One thread per
// (item, float4 slice).
__global__ void __launch_bounds__(256) seq_item_merge_kernel(SeqArgs s) {
  const SgdArgs& a = s.a;
  const int32_t K4 = a.K >> 2;
  const int64_t n = (int64_t)s.n_items * K4;
  const int64_t slot4 = a.n_rows * K4;
  const float4* base = reinterpret_cast<const float4*>(a.ring) + (int64_t)a.slot_base * slot4 +
                       (int64_t)a.n_users * K4;
  float4* out = reinterpret_cast<float4*>(a.ring) + (int64_t)a.slot_out * slot4 + (int64_t)a.n_users * K4;
  const float4* mine = reinterpret_cast<const float4*>(s.mine);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) {
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int32_t p = 0; p < s.P; ++p) {
      const float4 m = __ldg(mine + (int64_t)p * n + x);
      sum = make_float4(sum.x + m.x, sum.y + m.y, sum.z + m.z, sum.w + m.w);
    }
    const int32_t entries = __ldg(s.item_cnt + x / K4);
    if (entries > 0 && x % K4 == 0) s.chg_item[x / K4] = a.clock;
    const float sc = seq_cap_scale(a.cap, entries);
    const float4 b = base[x];
    out[x] = make_float4(b.x + sc * sum.x, b.y + sc * sum.y, b.z + sc * sum.z, b.w + sc * sum.w);
  }
}

}  // namespace

cudaError_t launch_seq_clock(const SeqArgs& s, cudaStream_t st) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const unsigned copiers = (unsigned)std::max<int64_t>(1, std::min<int64_t>((s.a.n_users + 63) / 64, (int64_t)sms * 8));
  auto go = [&](auto g, auto nv) {
    seq_users_kernel<decltype(g)::value, decltype(nv)::value><<<(unsigned)s.P + copiers, 64, 0, st>>>(s);
    return cudaGetLastError();
  };
  using std::integral_constant;
  const int32_t K4 = s.a.K >> 2;
  cudaError_t e;
  if (K4 <= 4) {
    e = go(integral_constant<int, 4>{}, integral_constant<int, 1>{});
  } else if (K4 <= 8) {
    e = go(integral_constant<int, 8>{}, integral_constant<int, 1>{});
  } else if (K4 <= 16) {
    e = go(integral_constant<int, 8>{}, integral_constant<int, 2>{});
  } else if (K4 <= 32) {
    e = K4 <= 24 ? go(integral_constant<int, 8>{}, integral_constant<int, 3>{})
                 : go(integral_constant<int, 8>{}, integral_constant<int, 4>{});
  } else if (K4 <= 64) {
    e = K4 <= 48 ? go(integral_constant<int, 16>{}, integral_constant<int, 3>{})
                 : go(integral_constant<int, 16>{}, integral_constant<int, 4>{});
  } else {
    e = K4 <= 96 ? go(integral_constant<int, 32>{}, integral_constant<int, 3>{})
                 : go(integral_constant<int, 32>{}, integral_constant<int, 4>{});
  }
  if (e != cudaSuccess) return e;
  const int64_t n = (int64_t)s.n_items * K4;
  if (n > 0) {
    const int mb = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sms * 8));
    seq_item_merge_kernel<<<mb, 256, 0, st>>>(s);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace esspt
