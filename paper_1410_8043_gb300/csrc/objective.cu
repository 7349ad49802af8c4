// The training objective (Sec. 3.1, Sec. 5) over all entries at one table
// version: sum e^2 and sum [e^2 + lambda (|L_i|^2 + |R_j|^2)], fp32 residuals
// and row norms, fp64 sums over the work items; whole, or by worker.
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
// The squares of U entries are added in fp32, their sums with the rounding error
// kept beside them (two-sum, Knuth, TAOCP vol. 2, 4.2.2): as good as adding each
// entry in fp64, whose units are few, since an entry's fp32 residual carries
// more error than U - 1 additions.  On the 20M entries, K = 100: 0.75 ms with
// plain fp32 sums per item (4.5e-9 off by worker where this is 5e-10), 1.09 ms
// with a two-sum per entry.
struct Sum2 {  // two packed fp32 sums and what they lost
  u64 sum = 0ull, lost = 0ull;
  __device__ __forceinline__ void add(u64 x, u64 minus1) {
    const u64 s = add2(sum, x), b = fma2(sum, minus1, s);                // b: the part of s that x became
    const u64 d = add2(fma2(fma2(b, minus1, s), minus1, sum), fma2(b, minus1, x));  // (sum - (s - b)) + (x - b)
    sum = s;
    lost = add2(lost, d);
  }
  __device__ __forceinline__ double total() const {
    float a, b, c, d;
    unpack2(sum, a, b);
    unpack2(lost, c, d);
    return ((double)a + (double)c) + ((double)b + (double)d);
  }
};

template <int G, int NV, bool BY_WORKER>
__global__ void __launch_bounds__(256) objective_kernel(ObjectiveArgs a) {
  constexpr int kGpw = 32 / G, U = NV == 1 ? 8 : NV == 2 ? 4 : 2;
  extern __shared__ double sums[];  // BY_WORKER: sum e^2 at [p], penalised sum at [P + p]
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
  const int64_t step = (((int64_t)gridDim.x * blockDim.x) >> 5) * kGpw;
  const u64 minus1 = pack2(-1.f, -1.f);
  double s1 = 0.0, s2 = 0.0;
  for (int64_t x0 = __ldg(a.item_base + blockIdx.y) + (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kGpw;
       x0 < x_end; x0 += step) {
    const int4 it = x0 + grp < x_end ? __ldg(a.items + x0 + grp) : make_int4(0, 0, 0, 0);
    const int32_t n = it.w >> 16, most = __reduce_max_sync(0xffffffffu, n);
    f2x2 L[NV];
    u64 l2 = 0ull;  // packed partial sums of |L|^2
    Sum2 r2, sq;    // of the entries' |R|^2; of e^2
#pragma unroll
    for (int k = 0; k < NV; ++k) {
      L[k] = f2x2{0ull, 0ull};
      ldg_f2x2_if(L[k], L4 + (int64_t)it.x * K4 + k * G, n > 0 && (k < NV - 1 || last_on));
      l2 = fma2(L[k].lo, L[k].lo, l2);
      l2 = fma2(L[k].hi, L[k].hi, l2);
    }
    for (int32_t t = 0; t < most; t += U) {
      f2x2 R[U][NV];
      float d[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const bool on = t + u < n;
        d[u] = on ? __ldg(rec_D + it.y + t + u) : 0.f;
        const int64_t j = on ? __ldg(rec_j + it.y + t + u) : 0;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          R[u][k] = f2x2{0ull, 0ull};
          ldg_f2x2_if(R[u][k], R4 + j * K4 + k * G, on && (k < NV - 1 || last_on));
        }
      }
      float dot[U];
      u64 rr[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        u64 p = 0ull;
        rr[u] = 0ull;
#pragma unroll
        for (int k = 0; k < NV; ++k) {
          p = fma2(L[k].lo, R[u][k].lo, p);
          p = fma2(L[k].hi, R[u][k].hi, p);
          rr[u] = fma2(R[u][k].lo, R[u][k].lo, rr[u]);
          rr[u] = fma2(R[u][k].hi, R[u][k].hi, rr[u]);
        }
        dot[u] = sum2(p);
      }
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1)
#pragma unroll
        for (int u = 0; u < U; ++u) dot[u] += __shfl_xor_sync(0xffffffffu, dot[u], off);
      float se = 0.f;
      u64 sr = 0ull;
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (t + u < n) {
          const float e = d[u] - dot[u];
          se = fmaf(e, e, se);
          sr = add2(sr, rr[u]);
        }
      sq.add(pack2(se, 0.f), minus1);
      r2.add(sr, minus1);
    }
    if (BY_WORKER) {
      double norm = n > 0 ? (double)n * (double)sum2(l2) + r2.total() : 0.0;
#pragma unroll
      for (int off = G / 2; off > 0; off >>= 1) norm += __shfl_xor_sync(0xffffffffu, norm, off);
      if (glane == 0 && n > 0) {
        const int p = it.w & 0xffff;
        atomicAdd(&sums[p], sq.total());
        atomicAdd(&sums[a.P + p], sq.total() + (double)a.lambda * norm);
      }
    } else if (n > 0) {
      s1 += glane == 0 ? sq.total() : 0.0;
      s2 += (double)n * (double)sum2(l2) + r2.total();
    }
  }
  if (BY_WORKER) {
    __syncthreads();
    for (int k = threadIdx.x; k < a.P; k += blockDim.x) {
      if (sums[k] != 0.0) atomicAdd(a.out + k, sums[k]);
      if (sums[a.P + k] != 0.0) atomicAdd(a.out + a.out_stride + k, sums[a.P + k]);
    }
  } else {
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
cudaError_t run(const ObjectiveArgs& a, cudaStream_t st) {
  auto go = [&](auto g, auto nv) {
    constexpr int G = decltype(g)::value, NV = decltype(nv)::value;
    const size_t smem = BY_WORKER ? 2 * sizeof(double) * (size_t)a.P : 0;
    int dev = 0, sms = 0, per_sm = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e == cudaSuccess)
      e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, objective_kernel<G, NV, BY_WORKER>, 256, smem);
    if (e != cudaSuccess) return e;
    // Two waves of blocks over the minibatches, no more than their items need.
    const int64_t need = (a.n_items / a.F + 8 * (32 / G)) / (8 * (32 / G));
    const int64_t x = std::max<int64_t>(1, std::min<int64_t>(need, 2ll * sms * per_sm / a.F));
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
