// The stream of a minibatch (see StreamArgs): its build when the data are
// loaded, new values for a staged minibatch, and the row-granular model's
// refresh, which writes a clock's x words.
#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace esspt {

// Warp w of n_warps takes items [part[w].x, part[w].y), the shares balanced by
// cost: pre[x] is the summed cost of the items before x (over all minibatches).
// They are whole rounds but for the minibatch's last, so that the empty places of
// partial rounds do not add up over the warps; one round each where that is all.
__global__ void __launch_bounds__(256) stream_partition_kernel(const int64_t* __restrict__ pre, int32_t n_items,
                                                               int32_t n_warps, int32_t gpw,
                                                               int4* __restrict__ part) {
  const int32_t w = blockIdx.x * blockDim.x + threadIdx.x;
  if (w > n_warps) return;
  int32_t lo = 0, hi = n_items;
  if (w == n_warps) {
    lo = n_items;
  } else if ((int64_t)n_warps * gpw >= n_items) {
    lo = w * gpw;
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
    lo = (int32_t)min((int64_t)n_items, ((int64_t)lo + gpw / 2) / gpw * gpw);
  }
  if (w < n_warps) part[w].x = lo;
  if (w > 0) part[w - 1].y = lo;
}

cudaError_t launch_stream_partition(const int64_t* pre, int64_t n_items, int64_t n_warps, const StreamGeometry& g,
                                    int4* part, cudaStream_t st) {
  stream_partition_kernel<<<(unsigned)(n_warps / 256 + 1), 256, 0, st>>>(pre, (int32_t)n_items, (int32_t)n_warps,
                                                                        g.gpw, part);
  return cudaGetLastError();
}

// Steps of every warp of a minibatch, in part[w].z for now.
__global__ void __launch_bounds__(256) stream_steps_kernel(const int4* __restrict__ items, int4* part,
                                                           int64_t n_warps, StreamGeometry g) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n_warps) return;
  const int lane = threadIdx.x & 31;
  const int32_t x0 = part[w].x, x1 = part[w].y;
  uint32_t sum = 0;
  for (int32_t r = x0 + lane * g.gpw; r < x1; r += 32 * g.gpw) {
    int32_t mx = 0;
    for (int32_t x = r; x < min(r + g.gpw, x1); ++x) mx = max(mx, items[x].w >> 16);
    sum += (mx + g.per_step - 1) / g.per_step;
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  if (lane == 0) part[w].z = (int32_t)sum;
}
// part[w].z, .w = first and end step of warp w; a warp starts at a multiple of
// kStepAlign steps, so that its records start on 16 bytes.  One block.
__global__ void __launch_bounds__(1024) stream_offsets_kernel(int4* part, int64_t n_warps, int64_t* total) {
  __shared__ int64_t sums[1024];
  const int64_t per = (n_warps + 1023) / 1024, w0 = threadIdx.x * per, w1 = min(n_warps, w0 + per);
  auto aligned = [&](int64_t w) {
    return ((int64_t)(uint32_t)part[w].z + kStepAlign - 1) / kStepAlign * kStepAlign;
  };
  int64_t sum = 0;
  for (int64_t w = w0; w < w1; ++w) sum += aligned(w);
  sums[threadIdx.x] = sum;
  __syncthreads();
  for (int off = 1; off < 1024; off <<= 1) {
    const int64_t v = threadIdx.x >= off ? sums[threadIdx.x - off] : 0;
    __syncthreads();
    sums[threadIdx.x] += v;
    __syncthreads();
  }
  int64_t at = sums[threadIdx.x] - sum;
  for (int64_t w = w0; w < w1; ++w) {
    const int64_t n = (uint32_t)part[w].z, next = at + aligned(w);
    part[w].z = (int32_t)(uint32_t)at;
    part[w].w = (int32_t)(uint32_t)(at + n);
    at = next;
  }
  if (threadIdx.x == 1023) *total = sums[1023];
}

cudaError_t launch_stream_steps(const int4* items, int4* part, int64_t n_warps, const StreamGeometry& g,
                                int64_t* total, cudaStream_t st) {
  stream_steps_kernel<<<(unsigned)(n_warps / 8 + 1), 256, 0, st>>>(items, part, n_warps, g);
  stream_offsets_kernel<<<1, 1024, 0, st>>>(part, n_warps, total);
  return cudaGetLastError();
}

// The records of a minibatch (x and yz hold kNoRecord everywhere on entry) and
// the place of every item's first entry.  One warp per warp of the kernel.
__global__ void __launch_bounds__(256) stream_fill_kernel(const int4* __restrict__ items,
                                                          const int4* __restrict__ part, int64_t n_warps,
                                                          StreamGeometry g, StreamSource src, uint32_t* __restrict__ x,
                                                          uint32_t* __restrict__ yz, uint32_t* __restrict__ place) {
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n_warps) return;
  const int lane = threadIdx.x & 31, G = 32 / g.gpw, grp = lane / G, l = lane & (G - 1);
  const int4 p = part[w];
  int64_t s = (uint32_t)p.z;
  for (int32_t x0 = p.x; x0 < p.y; x0 += g.gpw) {
    const int32_t i = x0 + grp;
    const int4 it = i < p.y ? items[i] : make_int4(0, 0, -2, 0);
    const int32_t n = it.w >> 16;
    const uint32_t at = place_word(g, s, grp);
    if (l == 0 && n > 0) place[i] = at;
    for (int32_t k = l; k < n; k += G) {
      const int32_t t = it.y + k, j = src.rec_j[t];
      const int32_t e0 = src.item_rep[j], e1 = src.item_rep[j + 1];  // extra replicas of j: e1 - e0 (reps - 1)
      const int32_t q = t & (e1 - e0);                               // reps is a power of two
      uint32_t y = (uint32_t)(q == 0 ? j : src.n_items + e0 + q - 1) * (uint32_t)src.dR_ld;
      if (src.hot_item != nullptr)
        for (int h = 0; h < kHot; ++h)
          if (src.hot_item[h] == j) y = 2u * h + 1u;
      const int64_t to = record_place(g, at, k);
      x[to] = (uint32_t)j * (uint32_t)(src.K / 4);
      yz[y_word(g, to)] = y;
      yz[y_word(g, to) + g.per_step] = __float_as_uint(src.rec_D[t]);
    }
    s += __reduce_max_sync(0xffffffffu, (n + g.per_step - 1) / g.per_step);
  }
}
cudaError_t launch_stream_fill(const int4* items, const int4* part, int64_t n_warps, const StreamGeometry& g,
                               const StreamSource& src, int64_t n_places, uint32_t* x, uint32_t* yz, uint32_t* place,
                               cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(x, 0xff, sizeof(uint32_t) * n_places, st);
  if (e == cudaSuccess) e = cudaMemsetAsync(yz, 0xff, 2 * sizeof(uint32_t) * n_places, st);
  if (e != cudaSuccess || n_warps <= 0) return e;
  stream_fill_kernel<<<(unsigned)((n_warps + 7) / 8), 256, 0, st>>>(items, part, n_warps, g, src, x, yz, place);
  return cudaGetLastError();
}

// New values of a minibatch's records: eight lanes per item.
__global__ void __launch_bounds__(256) stream_refill_kernel(const int4* __restrict__ items,
                                                            const uint32_t* __restrict__ place, int64_t n_items,
                                                            StreamGeometry g, const float* __restrict__ D,
                                                            uint32_t* __restrict__ yz) {
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; i < n_items; i += stride) {
    const int4 it = items[i];
    const uint32_t at = place[i];
    for (int32_t k = threadIdx.x & 7; k < it.w >> 16; k += 8)
      yz[y_word(g, record_place(g, at, k)) + g.per_step] = __float_as_uint(D[it.y + k]);
  }
}

cudaError_t launch_stream_refill(const int4* items, const uint32_t* place, int64_t n_items, const StreamGeometry& g,
                                 const float* D, uint32_t* yz, cudaStream_t st) {
  if (n_items <= 0) return cudaSuccess;
  stream_refill_kernel<<<grid_for(n_items, 32, 8), 256, 0, st>>>(items, place, n_items, g, D, yz);
  return cudaGetLastError();
}

// Row-granular SSP (Sec. 4 client cache, a clock c_param per cached row): for
// every work item, refresh its user's row and its entries' item rows in the
// cache of the reading worker; eight lanes per item.  All lanes that refresh
// one (worker, row) in a clock write the same value, c-1, so the races are
// benign and every read of the row in the clock sees one version.
__global__ void __launch_bounds__(256) row_refresh_kernel(RowRefreshArgs a) {
  const int32_t lo = a.c - 1 - a.s;
  const int64_t stride = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; i < a.n_items; i += stride) {
    const int4 it = __ldg(a.items + i);
    const uint32_t at = __ldg(a.place + i);
    int32_t* V = a.rowver + (int64_t)(it.w & 0xffff) * a.n_rows;
    if ((threadIdx.x & 7) == 0) {
      int32_t v = V[it.x];
      if (v < 0 || v < lo) {
        v = a.c - 1;
        V[it.x] = v;
      }
      a.user_slot[it.x] = v % a.nslots;
    }
    for (int32_t k = threadIdx.x & 7; k < it.w >> 16; k += 8) {
      const int64_t r = (int64_t)a.n_users + __ldg(a.rec_j + it.y + k);
      int32_t v = V[r];
      if (v < 0 || v < lo) {
        v = a.c - 1;
        V[r] = v;
      }
      a.x[record_place(a.g, at, k)] = (uint32_t)(((int64_t)(v % a.nslots) * a.n_rows + r) * a.K4);
    }
  }
}

cudaError_t launch_row_refresh(const RowRefreshArgs& a, cudaStream_t st) {
  if (a.n_items <= 0) return cudaSuccess;
  row_refresh_kernel<<<grid_for(a.n_items, 32, 8), 256, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace esspt
