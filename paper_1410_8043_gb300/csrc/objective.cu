// The training objective (Sec. 3.1, Sec. 5) over all entries at one table
// version: sum e^2 and sum [e^2 + lambda (|L_i|^2 + |R_j|^2)], fp32 residuals
// and row norms, summed to the precision of fp64; whole, or by worker.
#include <algorithm>
#include <type_traits>

#include "internal.h"
#include "ptx.cuh"

namespace esspt {

namespace {

// The work list of every minibatch (blockIdx.y): row groups of G lanes (NV
// float4 slices of a row per lane, G (NV - 1) < K/4 <= G NV), one item each, the groups of a warp side by
// side on items of (nearly) one length.  L stays in registers over an item's
// entries and |L|^2 is taken once per item, so an entry costs one gathered row;
// U of them are in flight per group.  What bounds it is those gathers (K = 100:
// 400 bytes per entry out of L2).  One warp per entry, which it replaces, read
// both rows and reduced three sums per entry: 11.0 ms on 20M entries, K = 100.
//
// Every entry's exact square (high and low fp32 parts) is added to an fp32 sum
// with its rounding error kept beside it (two-sum, Knuth, TAOCP vol. 2, 4.2.2);
// fp64, whose units are few, only at the end: an fp64 sum per item takes 1.05 ms
// on those 20M entries, this 0.77.  Squares added eight at a time without their
// rounding errors were 8.7e-10 off on 51k entries, the exact ones 7e-11.  What
// fp32 cannot hold so goes to fp64 sums of its own: squares and norms from 1e29
// on, NaN among them (a lane adds fewer than 2^31 of them, which stay finite
// below it), and squares whose low part would be subnormal.
constexpr float kHuge = 1e29f;
__device__ __forceinline__ bool in_range(float e, float norm) {
  return fabsf(e) < 3e14f && !(fabsf(e) < 1e-14f && e != 0.f) && norm < kHuge;
}
// Rows of a group in flight.
template <int G, int NV>
constexpr int kInFlight = NV >= 3 ? 2 : NV == 2 || G == 4 ? 4 : 8;
constexpr int32_t kPart = 8;  // entries of a part of an item at most
// x + y and its rounding error.
__device__ __forceinline__ float two_sum(float x, float y, float& err) {
  const float s = x + y, b = s - x;
  err = (x - (s - b)) + (y - b);
  return s;
}
struct Sum2 {  // two packed fp32 sums and what they lost
  u64 sum = 0ull, lost = 0ull;
  __device__ __forceinline__ void add(u64 x, u64 minus1) {
    const u64 s = add2(sum, x), b = fma2(sum, minus1, s);                // b: the part of s that x became
    const u64 d = add2(fma2(fma2(b, minus1, s), minus1, sum), fma2(b, minus1, x));  // (sum - (s - b)) + (x - b)
    sum = s;
    lost = add2(lost, d);
  }
};

// Four blocks per SM, as the grid is sized for, where that spills nothing.  1.5M
// entries, us: K = 512 286 with what the compiler takes (66..72 registers), 228 so.
// By worker at K = 100..128 three (1.5M entries, K = 128: 141 with four, 110).
template <int G, int NV, bool BY_WORKER>
__global__ void __launch_bounds__(256, G == 8 && (NV == 1 || (BY_WORKER && NV == 4)) ? 3 : 4)
    objective_kernel(ObjectiveArgs a) {
  constexpr int kGpw = 32 / G, U = kInFlight<G, NV>;
  extern __shared__ double sums[];  // BY_WORKER: sum e^2 at [p], of the rows' squares at [P + p]
  if (BY_WORKER) {
    for (int k = threadIdx.x; k < 2 * a.P; k += blockDim.x) sums[k] = 0.0;
    __syncthreads();
  }
  const int lane = threadIdx.x & 31, glane = lane & (G - 1), grp = lane / G;
  const int32_t K4 = a.K >> 2;
  const bool last_on = glane + (NV - 1) * G < K4;
  const float4* L4 = reinterpret_cast<const float4*>(a.slot) + glane;
  const float4* R4 = L4 + a.n_users * K4;
  const int64_t x_end = __ldg(a.item_base + blockIdx.y + 1), e_base = __ldg(a.entry_base + blockIdx.y);
  const int32_t* rec_j = a.rec_j + e_base;
  const float* rec_D = a.rec_D + e_base;
  const uint32_t step = (gridDim.x * blockDim.x) >> 5;
  const u64 minus1 = pack2(-1.f, -1.f);
  // e^2 and what the rows' squares add up to; by worker, of the item at hand.
  Sum2 sums2;  // (e^2, this lane's part of the rows' squares)
  double wide_e = 0.0, wide_n = 0.0;  // the same of what fp32 cannot hold, and whether there is any
  bool wide = false;
  // BY_WORKER: the sums of the group's last items, one per lane: the fp64 units are
  // as long with an instruction for one lane as for all (190k entries, one or two
  // per item, K = 496: 200 us with fp64 sums for each item in turn, 133 so).
  float kept_e = 0.f, kept_el = 0.f, kept_n = 0.f, kept_nl = 0.f;
  int kept_p = -1, kept = 0;
  auto flush = [&]() {
    const double sq = (double)kept_e + (double)kept_el, norms = (double)kept_n + (double)kept_nl;
    // Few places, which many lanes would add to in turn: one addition per worker (the
    // same case with 1, 2 and 3 workers: 203, 176, 164 us without; 139, 152, 154; with
    // 8 workers 152, and 190 so).
    if (a.P <= 3) {
      for (unsigned left = __ballot_sync(0xffffffffu, kept_p >= 0); left != 0u;) {
        const int p = __shfl_sync(0xffffffffu, kept_p, __ffs(left) - 1);
        double x = kept_p == p ? sq : 0.0, y = kept_p == p ? norms : 0.0;
#pragma unroll 1
        for (int off = 16; off > 0; off >>= 1) {
          x += __shfl_xor_sync(0xffffffffu, x, off);
          y += __shfl_xor_sync(0xffffffffu, y, off);
        }
        if (lane == 0) {
          atomicAdd(&sums[p], x);
          atomicAdd(&sums[a.P + p], y);
        }
        left &= ~__ballot_sync(0xffffffffu, kept_p == p);
      }
    } else if (kept_p >= 0) {
      atomicAdd(&sums[kept_p], sq);
      atomicAdd(&sums[a.P + kept_p], norms);
    }
    kept_p = -1;
    kept = 0;
  };
  // Units of kGpw items, or of a part of each.
  const int64_t x_first = __ldg(a.item_base + blockIdx.y);
  const uint32_t units = (uint32_t)((x_end - x_first + kGpw - 1) / kGpw);
  for (uint32_t v = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < units * max(a.parts, 1); v += step) {
    const uint32_t part = a.parts > 0 ? v / units : 0;
    const int64_t x0 = x_first + (int64_t)(v - part * units) * kGpw;
    int4 it = x0 + grp < x_end ? __ldg(a.items + x0 + grp) : make_int4(0, 0, 0, 0);
    int32_t n = it.w >> 16;
    if (a.parts > 0) {
      it.y += part * a.part;
      n = min(max(n - (int32_t)part * a.part, 0), a.part);
    }
    const int32_t most = __reduce_max_sync(0xffffffffu, n);
    if (most == 0) continue;
    if (BY_WORKER) sums2 = Sum2{};
    int32_t lane_j = 0;  // the next G entries by lane
    float lane_d = 0.f;
    if (glane < n) {
      lane_j = __ldg(rec_j + it.y + glane);
      lane_d = __ldg(rec_D + it.y + glane);
    }
    f2x2 L[NV];
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      L[k] = f2x2{0ull, 0ull};
      ldg_f2x2_if(L[k], L4 + (int64_t)it.x * K4 + k * G, n > 0 && (k < NV - 1 || last_on));
    }
#pragma unroll 1
    for (int32_t t = 0; t < most; t += U) {
      // By lane, so that no step's rows wait for a load of ids (9M entries, K = 32 and
      // 64: 241 and 205 us with one load per step, 197 and 184 so).
      if (t > 0 && (t & (G - 1)) == 0 && t + glane < n) {
        lane_j = __ldg(rec_j + it.y + t + glane);
        lane_d = __ldg(rec_D + it.y + t + glane);
      }
      f2x2 R[U][NV];
      float d[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        d[u] = __shfl_sync(0xffffffffu, lane_d, t + u, G);
        const int64_t j = __shfl_sync(0xffffffffu, lane_j, t + u, G);
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          R[u][k] = f2x2{0ull, 0ull};
          ldg_f2x2_if(R[u][k], R4 + j * K4 + k * G, t + u < n && (k < NV - 1 || last_on));
        }
      }
      float e[U], norm[U];  // residuals, and this lane's part of |R|^2
#pragma unroll
      for (int u = 0; u < U; ++u) {
        u64 p = 0ull, r = 0ull;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          p = fma2(L[k].lo, R[u][k].lo, p);
          p = fma2(L[k].hi, R[u][k].hi, p);
          r = fma2(R[u][k].lo, R[u][k].lo, r);
          r = fma2(R[u][k].hi, R[u][k].hi, r);
        }
        e[u] = sum2(p);
        norm[u] = sum2(r);
      }
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) e[u] += __shfl_xor_sync(0xffffffffu, e[u], off);
      bool odd = false;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        e[u] = t + u < n ? d[u] - e[u] : 0.f;
        odd |= !in_range(e[u], norm[u]);
      }
      if (odd) {  // (one branch for the step: one per entry took 1380 us instead of 802, 20M entries, K = 100)
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (!in_range(e[u], norm[u])) {
            wide_e += (double)e[u] * (double)e[u];
            wide_n += (double)norm[u];
            e[u] = norm[u] = 0.f;
            wide = true;
          }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const float high = e[u] * e[u];
        sums2.add(pack2(high, norm[u]), minus1);
        sums2.lost = add2(sums2.lost, pack2(fmaf(e[u], e[u], -high), 0.f));
      }
    }
    if (n > 0) {
      u64 l2 = 0ull;
#pragma unroll
      for (int k = 0; k < NV; ++k) {
        l2 = fma2(L[k].lo, L[k].lo, l2);
        l2 = fma2(L[k].hi, L[k].hi, l2);
      }
      const float l = sum2(l2);
      float high = (float)n * l, low = fmaf((float)n, l, -high);
      if (!(high < kHuge)) {
        wide_n += (double)n * (double)l;
        high = low = 0.f;
        wide = true;
      }
      sums2.add(pack2(0.f, high), minus1);
      sums2.lost = add2(sums2.lost, pack2(0.f, low));
    }
    if (BY_WORKER) {
      float e2, e2_lost, norm, norm_lost;
      unpack2(sums2.sum, e2, norm);
      unpack2(sums2.lost, e2_lost, norm_lost);
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) {
        const float lost = __shfl_xor_sync(0xffffffffu, norm_lost, off);
        float err;
        norm = two_sum(norm, __shfl_xor_sync(0xffffffffu, norm, off), err);
        norm_lost += lost + err;
      }
      if (glane == kept && n > 0) {
        kept_e = e2;
        kept_el = e2_lost;
        kept_n = norm;
        kept_nl = norm_lost;
        kept_p = it.w & 0xffff;
      }
      if (++kept == G) flush();
      if (__any_sync(0xffffffffu, wide)) {
#pragma unroll 1
        for (int off = G / 2; off > 0; off >>= 1) wide_n += __shfl_xor_sync(0xffffffffu, wide_n, off);
        if (glane == 0 && n > 0) {
          atomicAdd(&sums[it.w & 0xffff], wide_e);
          atomicAdd(&sums[a.P + (it.w & 0xffff)], wide_n);
        }
        wide_e = wide_n = 0.0;
        wide = false;
      }
    }
  }
  if (BY_WORKER) {
    flush();
    __syncthreads();
    for (int k = threadIdx.x; k < a.P; k += blockDim.x) {
      const double sq = sums[k], pen = sq + (double)a.lambda * sums[a.P + k];
      if (sq != 0.0) atomicAdd(a.out + k, sq);
      if (pen != 0.0) atomicAdd(a.out + a.out_stride + k, pen);
    }
  } else {
    float e2, e2_lost, norm, norm_lost;
    unpack2(sums2.sum, e2, norm);
    unpack2(sums2.lost, e2_lost, norm_lost);
    double s1 = glane == 0 ? (double)e2 + (double)e2_lost + wide_e : 0.0;
    double s2 = (double)norm + (double)norm_lost + wide_n;
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, off);
      s2 += __shfl_xor_sync(0xffffffffu, s2, off);
    }
    __shared__ double part[2][8];
    if (lane == 0) {
      part[0][threadIdx.x >> 5] = s1;
      part[1][threadIdx.x >> 5] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double x = 0.0, y = 0.0;
      for (int w = 0; w < 8; ++w) {
        x += part[0][w];
        y += part[1][w];
      }
      atomicAdd(a.out, x);
      atomicAdd(a.out + a.out_stride, x + (double)a.lambda * y);
    }
  }
}

template <bool BY_WORKER>
cudaError_t run(ObjectiveArgs a, cudaStream_t st) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  auto go = [&](auto g, auto nv) {
    constexpr int G = decltype(g)::value, NV = decltype(nv)::value, kGpw = 32 / G;
    const size_t smem = BY_WORKER ? 2 * sizeof(double) * (size_t)a.P : 0;
    // With fewer items than the GPU holds groups, or some of them far longer than a
    // group's share of the entries, an item is taken in parts, so that a call lasts
    // no longer than the gathers of one part (20k entries, K = 224: 77 us whole, 41
    // in parts of 8; 13k entries in 8k items, some of 96, K = 512: 66 and 40).
    // A warp then looks at units * parts / resident units, most of them empty.  The
    // parts are of 2 entries where one look per warp takes them all, else of 4 or 8
    // (1k entries, K = 100: 13 us of kernel in parts of 8, 8 of 2).  Blocks (four per
    // SM) for about two waves over the minibatches where there is work for them, for
    // parts one: every block ends in two fp64 additions to one place (13k entries of
    // 531k users, K = 64: 41 us with two waves, 30 with one; half a wave 32).
    const int64_t resident = 4ll * sms * 8, groups = resident * kGpw, units = a.n_items / kGpw + a.F;
    auto parts_of = [&](int32_t part) { return (a.longest + part - 1) / part; };
    const int64_t share = a.n_obs / groups, steps = (std::max<int64_t>(a.longest, share) - share) / kInFlight<G, NV>;
    const bool in_parts = a.n_items < groups || units * parts_of(kPart) / resident < steps;
    a.part = 2;
    while (a.part < kPart && units * parts_of(a.part) > resident) a.part *= 2;
    a.parts = in_parts ? parts_of(a.part) : 0;
    const int64_t need = ((in_parts ? a.parts : 1) * (a.n_items / a.F + kGpw) / kGpw + 7) / 8, wave = resident / 8 / a.F;
    const int64_t x = std::max<int64_t>(1, std::min<int64_t>(need, in_parts || need < 4 * wave ? wave : 2 * wave));
    objective_kernel<G, NV, BY_WORKER><<<dim3((unsigned)x, (unsigned)a.F), 256, smem, st>>>(a);
    return cudaGetLastError();
  };
  using std::integral_constant;
  const int32_t K4 = a.K / 4;
  if (K4 <= 4) return go(integral_constant<int, 4>{}, integral_constant<int, 1>{});
  if (K4 <= 8) return go(integral_constant<int, 8>{}, integral_constant<int, 1>{});
  if (K4 <= 16) return go(integral_constant<int, 8>{}, integral_constant<int, 2>{});
  if (K4 <= 24) return go(integral_constant<int, 8>{}, integral_constant<int, 3>{});
  if (K4 <= 32) return go(integral_constant<int, 8>{}, integral_constant<int, 4>{});
  if (K4 <= 48) return go(integral_constant<int, 16>{}, integral_constant<int, 3>{});
  if (K4 <= 64) return go(integral_constant<int, 16>{}, integral_constant<int, 4>{});
  if (K4 <= 96) return go(integral_constant<int, 32>{}, integral_constant<int, 3>{});
  return go(integral_constant<int, 32>{}, integral_constant<int, 4>{});
}

}  // namespace

cudaError_t launch_objective(const ObjectiveArgs& a, cudaStream_t st) {
  const cudaError_t e = cudaMemsetAsync(a.out, 0, 2 * sizeof(double), st);
  return e != cudaSuccess || a.n_items == 0 ? e : run<false>(a, st);
}

cudaError_t launch_worker_objective(const ObjectiveArgs& a, cudaStream_t st) {
  return a.n_items == 0 ? cudaSuccess : run<true>(a, st);
}

}  // namespace esspt
