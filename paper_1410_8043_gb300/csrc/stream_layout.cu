// The stream of a minibatch (see StreamArgs): its build when the data are
// loaded, new values for a staged minibatch, and the row-granular model's
// refresh, which writes a clock's x words.
#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace esspt {

// Warps of a minibatch: at most one per round of its items.
__device__ __forceinline__ int64_t warps_of(const StreamBuild& b, int32_t f) {
  const int64_t items = __ldg(b.item_base + f + 1) - __ldg(b.item_base + f);
  return min(b.max_warps, (items + b.g.gpw - 1) / b.g.gpw);
}

// Warp w of minibatch blockIdx.y's takes items [part[w].x, part[w].y), the shares
// balanced by cost: pre[x] is the summed cost of the items before x (over all
// minibatches).  They are whole rounds but for the minibatch's last, so that the
// empty places of partial rounds do not add up over the warps; one round each
// where that is all.
__global__ void __launch_bounds__(256) stream_partition_kernel(StreamBuild b) {
  const int32_t f = blockIdx.y, gpw = b.g.gpw;
  __shared__ int64_t first;
  if (threadIdx.x == 0) {
    first = 0;
    for (int32_t k = 0; k < f; ++k) first += warps_of(b, k);
    if (blockIdx.x == 0) {
      b.part_base[f] = first;
      if (f == b.F - 1) b.part_base[b.F] = first + warps_of(b, f);
    }
  }
  __syncthreads();
  const int64_t x0 = __ldg(b.item_base + f), n_items = __ldg(b.item_base + f + 1) - x0, n_warps = warps_of(b, f);
  const int64_t* pre = b.pre + x0;
  int4* part = b.part + first;
  const int64_t w = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (w > n_warps) return;
  int64_t lo = 0, hi = n_items;
  if (w == n_warps) {
    lo = n_items;
  } else if (n_warps * gpw >= n_items) {
    lo = w * gpw;
  } else {
    const int64_t target = pre[0] + (int64_t)((double)(pre[n_items] - pre[0]) * w / n_warps);
    while (lo < hi) {
      const int64_t m = lo + (hi - lo) / 2;
      if (pre[m] >= target) {
        hi = m;
      } else {
        lo = m + 1;
      }
    }
    lo = min(n_items, (lo + gpw / 2) / gpw * gpw);
  }
  if (w < n_warps) part[w].x = (int32_t)lo;
  if (w > 0) part[w - 1].y = (int32_t)lo;
}

// Steps of every warp, in part[w].z for now.
__global__ void __launch_bounds__(256) stream_steps_kernel(StreamBuild b) {
  const int32_t f = blockIdx.y;
  const int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5, first = __ldg(b.part_base + f);
  if (w >= __ldg(b.part_base + f + 1) - first || (*b.status & kErrInput) != 0u) return;
  const int lane = threadIdx.x & 31;
  const int4* items = b.items + __ldg(b.item_base + f);
  int4* part = b.part + first + w;
  const int64_t x0 = part->x, x1 = part->y;
  uint32_t sum = 0;
  for (int64_t r = x0 + lane * b.g.gpw; r < x1; r += 32 * b.g.gpw) {
    int32_t mx = 0;
    for (int64_t x = r; x < min(r + b.g.gpw, x1); ++x) mx = max(mx, items[x].w >> 16);
    sum += (mx + b.g.per_step - 1) / b.g.per_step;
  }
  sum = __reduce_add_sync(0xffffffffu, sum);
  if (lane == 0) part->z = (int32_t)sum;
}

// part[w].z, .w = first and end step of warp w; a warp starts at a multiple of
// kStepAlign steps, so that its records start on 16 bytes.  One block per
// minibatch.
__global__ void __launch_bounds__(1024) stream_offsets_kernel(StreamBuild b) {
  __shared__ int64_t sums[1024];
  const int32_t f = blockIdx.x;
  int4* part = b.part + __ldg(b.part_base + f);
  const int64_t n_warps = __ldg(b.part_base + f + 1) - __ldg(b.part_base + f);
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
  if (threadIdx.x == 1023) b.steps[f] = sums[1023];
}

// The records of minibatch blockIdx.y, empty places among them, and the place of
// every item's first entry.  One warp per warp of the kernel.
__global__ void __launch_bounds__(256) stream_fill_kernel(StreamBuild b) {
  const int32_t f = blockIdx.y, K4 = b.K / 4;
  const StreamGeometry g = b.g;
  __shared__ int64_t first;
  if (threadIdx.x == 0) {
    first = 0;
    for (int32_t k = 0; k < f; ++k) first += __ldg(b.steps + k) * g.gpw * g.per_step;
    if (blockIdx.x == 0) {
      b.place_base[f] = first;
      if (f == b.F - 1) b.place_base[b.F] = first + __ldg(b.steps + f) * g.gpw * g.per_step;
    }
  }
  __syncthreads();
  const int64_t steps = __ldg(b.steps + f), w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= __ldg(b.part_base + f + 1) - __ldg(b.part_base + f)) return;
  if ((*b.status & kErrInput) != 0u || steps > kMaxSteps || first + steps * g.gpw * g.per_step > b.max_places) return;
  const int lane = threadIdx.x & 31, G = 32 / g.gpw, grp = lane / G, l = lane & (G - 1);
  const int64_t x_first = __ldg(b.item_base + f), e_first = __ldg(b.entry_base + f);
  const int4* items = b.items + x_first;
  const int32_t* rec_j = b.rec_j + e_first;
  const float* rec_D = b.rec_D + e_first;
  uint32_t *x = b.x + first, *yz = b.yz + 2 * first, *place = b.place + x_first;
  int32_t hot[kHot];
#pragma unroll
  for (int h = 0; h < kHot; ++h) hot[h] = b.hot_item != nullptr ? __ldg(b.hot_item + (int64_t)f * kHot + h) : -1;
  const int4 p = b.part[__ldg(b.part_base + f) + w];
  int64_t s = (uint32_t)p.z;
  for (int64_t x0 = p.x; x0 < p.y; x0 += g.gpw) {
    const int64_t i = x0 + grp;
    const int4 it = i < p.y ? items[i] : make_int4(0, 0, -2, 0);
    const int32_t n = it.w >> 16;
    const int32_t most = __reduce_max_sync(0xffffffffu, (n + g.per_step - 1) / g.per_step);
    const uint32_t at = place_word(g, s, grp);
    if (l == 0 && n > 0) place[i] = at;
    for (int32_t k = l; k < most * g.per_step; k += G) {
      uint32_t xw = kNoRecord, y = kNoRecord, z = kNoRecord;
      if (k < n) {
        const int32_t t = it.y + k, j = rec_j[t];
        const int32_t e0 = b.item_rep[j], e1 = b.item_rep[j + 1];  // extra replicas of j: e1 - e0 (reps - 1)
        const int32_t q = t & (e1 - e0);                           // reps is a power of two
        xw = (uint32_t)j * (uint32_t)K4;
        y = (uint32_t)(q == 0 ? j : b.n_items + e0 + q - 1) * (uint32_t)b.dR_ld;
#pragma unroll
        for (int h = 0; h < kHot; ++h)
          if (hot[h] == j) y = 2u * h + 1u;
        z = __float_as_uint(rec_D[t]);
      }
      const int64_t to = record_place(g, at, k), to_y = y_word(g, to);
      x[to] = xw;
      yz[to_y] = y;
      yz[to_y + g.per_step] = z;
    }
    s += most;
  }
}

cudaError_t launch_stream_build(const StreamBuild& b, cudaStream_t st) {
  const int64_t warps = std::min(b.max_warps, (b.max_items + b.g.gpw - 1) / b.g.gpw);
  const unsigned F = (unsigned)b.F;
  stream_partition_kernel<<<dim3((unsigned)(warps / 256 + 1), F), 256, 0, st>>>(b);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  stream_steps_kernel<<<dim3((unsigned)(warps / 8 + 1), F), 256, 0, st>>>(b);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  stream_offsets_kernel<<<F, 1024, 0, st>>>(b);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  stream_fill_kernel<<<dim3((unsigned)(warps / 8 + 1), F), 256, 0, st>>>(b);
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
