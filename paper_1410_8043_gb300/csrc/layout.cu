// Setup (once per data set, not per clock): lay the observed entries out by
// minibatch and user so that a clock streams one contiguous, user-sorted
// segment (Sec. 3.1: D_obs partitioned over workers; Sec. 5: a fixed
// minibatch per Clock()).  The radix sort is stable, so entries of a user
// keep their input order and every run sees the same layout.  Also builds
// the chunk and heavy-user lists and the replica rows of popular items and
// heavy users.
#include <algorithm>
#include <vector>

#include <cub/device/device_radix_sort.cuh>
#include <cub/device/device_scan.cuh>
#include <thrust/iterator/counting_iterator.h>
#include <thrust/iterator/transform_iterator.h>

#include "internal.h"

namespace esspt {

namespace {

inline size_t align256(size_t x) { return (x + 255) & ~size_t(255); }

__host__ __device__ inline int32_t next_pow2(int32_t x) {
  int32_t p = 1;
  while (p < x) p <<= 1;
  return p;
}

// Replicas of a heavy user with nch chunks: one per kUserRep chunks, rounded
// up to a power of two (never more than nch), at most kMaxRep.
__host__ __device__ inline int32_t user_reps(int32_t nch) {
  const int32_t r = next_pow2((nch + kUserRep - 1) / kUserRep);
  return r < kMaxRep ? r : kMaxRep;
}

// Replicas of an item whose largest minibatch count is mx, at most kMaxRep.
__host__ __device__ inline int32_t item_reps(int32_t mx) {
  const int32_t want = (mx + kItemRep - 1) / kItemRep;
  const int32_t r = next_pow2(want > 1 ? want : 1);
  return r < kMaxRep ? r : kMaxRep;
}

__global__ void validate_kernel(const int32_t* __restrict__ i, const int32_t* __restrict__ j,
                                const uint8_t* __restrict__ mb, int64_t n_obs, const int32_t* __restrict__ worker,
                                int64_t n_users, int64_t n_items, int32_t F, int32_t P, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_obs; k += stride)
    bad |= i[k] < 0 || i[k] >= n_users || j[k] < 0 || j[k] >= n_items || mb[k] >= F;
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n_users; u += stride)
    bad |= worker[u] < 0 || worker[u] >= P;
  if (bad) atomicOr(status, kErrInput);
}

__global__ void keys_kernel(const int32_t* __restrict__ i, const int32_t* __restrict__ j,
                            const uint8_t* __restrict__ mb, int64_t n_obs, int64_t n_users, int64_t n_items,
                            uint32_t* __restrict__ key, uint32_t* __restrict__ val, int32_t* __restrict__ cnt,
                            int32_t* __restrict__ item_cnt) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_obs; k += stride) {
    const uint32_t x = (uint32_t)((int64_t)mb[k] * n_users + i[k]);
    key[k] = x;
    val[k] = (uint32_t)k;
    atomicAdd(cnt + x, 1);
    atomicAdd(item_cnt + (int64_t)mb[k] * n_items + j[k], 1);
  }
}

__global__ void gather_kernel(const uint32_t* __restrict__ perm, int64_t n_obs, const int32_t* __restrict__ i,
                              const int32_t* __restrict__ j, const float* __restrict__ D, int32_t* __restrict__ ru,
                              int32_t* __restrict__ rj, float* __restrict__ rD) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n_obs; k += stride) {
    const uint32_t s = perm[k];
    ru[k] = i[s];
    rj[k] = j[s];
    rD[k] = D[s];
  }
}

// uoff[b][u] = off[b*N+u] - off[b*N] for u in [0, N]; mb_base[b] = off[b*N];
// per (b, u): chunks, heavy flag and extra replica rows.
__global__ void offsets_kernel(const int64_t* __restrict__ off, int64_t n_users, int32_t F, int32_t* __restrict__ uoff,
                               int64_t* __restrict__ mb_base, const int32_t* __restrict__ cnt,
                               int32_t* __restrict__ nch, int32_t* __restrict__ hflag, int32_t* __restrict__ hextra) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t total = (int64_t)F * (n_users + 1);
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += stride) {
    const int64_t b = x / (n_users + 1), u = x % (n_users + 1);
    const int64_t base = off[b * n_users];
    uoff[x] = (int32_t)(off[b * n_users + u] - base);
    if (u == 0) mb_base[b] = base;
    if (u < n_users) {
      const int32_t n = cnt[b * n_users + u];
      const int32_t c = n > kHeavy ? (n + kChunk - 1) / kChunk : 0;
      nch[b * n_users + u] = c + (n > 0 && c == 0 ? 1 : 0);
      hflag[b * n_users + u] = c > 0 ? 1 : 0;
      hextra[b * n_users + u] = c > 0 ? user_reps(c) - 1 : 0;
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) mb_base[F] = off[(int64_t)F * n_users];
}

// Work items (see StreamArgs) and heavy-user descriptors (user, first extra
// replica row, replicas, entries).  Replica 0 of heavy user u is row u of dL;
// replicas 1.. are rows n_users + hext[...].
__global__ void heavy_kernel(const int64_t* __restrict__ choff, const int32_t* __restrict__ nch,
                             const int64_t* __restrict__ hoff, const int64_t* __restrict__ hext,
                             const int32_t* __restrict__ uoff, const int32_t* __restrict__ worker, int64_t n_users,
                             int32_t F, int4* __restrict__ chunk,
                             uint32_t* __restrict__ key, uint32_t* __restrict__ val, int64_t n_tiles,
                             int64_t* __restrict__ chunk_base, int64_t max_chunks, int4* __restrict__ heavy,
                             int64_t* __restrict__ heavy_base, int64_t max_heavy, int64_t max_user_reps,
                             uint32_t* longest, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t total = (int64_t)F * n_users;
  int32_t most = 0;
  auto put = [&](int64_t at, int64_t b, int64_t u, int32_t beg, int32_t dst, int32_t n) {
    most = max(most, n);
    chunk[at] = make_int4((int32_t)u, beg, dst, n << 16 | worker[u]);
    key[at] = (uint32_t)(b * n_tiles + (u >> kTileBits)) << 7 | (uint32_t)(127 - n);
    val[at] = (uint32_t)at;
  };
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < total; x += stride) {
    const int32_t nc = nch[x];
    if (nc == 0) continue;
    const int64_t b = x / n_users, u = x % n_users;
    const int32_t beg = uoff[b * (n_users + 1) + u], end = uoff[b * (n_users + 1) + u + 1];
    if (end - beg <= kHeavy) {  // a light user: one work item, written directly
      if (choff[x] >= max_chunks) {
        atomicOr(status, kErrInput);
        continue;
      }
      put(choff[x], b, u, beg, -1, end - beg);
      continue;
    }
    const int32_t reps = user_reps(nc);
    const int64_t extra0 = n_users + hext[x];
    // The bounds below hold by construction; the checks keep every store in range.
    if (hoff[x] >= max_heavy || choff[x] + nc > max_chunks || hext[x] + reps - 1 > max_user_reps) {
      atomicOr(status, kErrInput);
      continue;
    }
    heavy[hoff[x]] = make_int4((int32_t)u, (int32_t)extra0, reps, end - beg);
    for (int32_t t = 0; t < nc; ++t) {
      const int32_t r = t & (reps - 1);
      const int32_t dst = r == 0 ? (int32_t)u : (int32_t)(extra0 + r - 1);
      put(choff[x] + t, b, u, beg + t * kChunk, dst, min(kChunk, end - beg - t * kChunk));
    }
  }
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= F; b += stride) {
    chunk_base[b] = choff[b * n_users];
    heavy_base[b] = hoff[b * n_users];
  }
  most = __reduce_max_sync(0xffffffffu, most);
  if ((threadIdx.x & 31) == 0 && most > 0) atomicMax(longest, (uint32_t)most);
}

// Extra replica rows of every item (replicas - 1) from its largest minibatch
// count.  Replica 0 of item j is row j of dR; the extra ones follow all items.
__global__ void item_reps_kernel(const int32_t* __restrict__ item_cnt, int64_t n_items, int32_t F,
                                 int32_t* __restrict__ reps) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j <= n_items; j += stride) {
    if (j == n_items) {
      reps[j] = 0;
      continue;
    }
    int32_t mx = 0;
    for (int32_t b = 0; b < F; ++b) mx = max(mx, item_cnt[(int64_t)b * n_items + j]);
    reps[j] = item_reps(mx) - 1;
  }
}

// wbase[p] = first place of worker p among the sorted workers of the users.
__global__ void worker_bases_kernel(const uint32_t* __restrict__ sorted, int64_t n_users, int32_t P,
                                    int32_t* __restrict__ wbase) {
  const int32_t p = blockIdx.x * blockDim.x + threadIdx.x;
  if (p > P) return;
  int64_t lo = 0, hi = n_users;
  while (lo < hi) {
    const int64_t m = (lo + hi) / 2;
    if (sorted[m] >= (uint32_t)p) {
      hi = m;
    } else {
      lo = m + 1;
    }
  }
  wbase[p] = (int32_t)lo;
}

__global__ void iota_kernel(uint32_t* __restrict__ val, int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride) val[k] = (uint32_t)k;
}

// The work list in its final order.
__global__ void place_items_kernel(const int4* __restrict__ raw, const uint32_t* __restrict__ perm, int64_t n,
                                   int4* __restrict__ items) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t x = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; x < n; x += stride) items[x] = raw[perm[x]];
}

// Cost of item x (64 bits: a scan adds in its input's type, and the costs of a
// data set pass 2^31); 0 past the last.
struct ItemCost {
  const int4* items;
  int64_t n;
  __host__ __device__ int64_t operator()(int64_t x) const { return x < n ? (items[x].w >> 16) + kItemCost : 0; }
};
cudaError_t scan_costs(void* tmp, size_t& bytes, const int4* items, int64_t n, int64_t* pre, cudaStream_t st) {
  const auto cost = thrust::make_transform_iterator(thrust::counting_iterator<int64_t>(0), ItemCost{items, n});
  return cub::DeviceScan::ExclusiveSum(tmp, bytes, cost, pre, (int)(n + 1), st);
}

// The items with extra replicas.
__global__ void popular_kernel(const int32_t* __restrict__ item_rep, int64_t n_items, int64_t max_popular,
                               int4* __restrict__ popular, uint32_t* __restrict__ n_popular, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < n_items; j += stride) {
    const int32_t e0 = item_rep[j], extra = item_rep[j + 1] - e0;
    if (extra == 0) continue;
    const uint32_t at = atomicAdd(n_popular, 1u);
    if (at < max_popular) {
      popular[at] = make_int4((int32_t)j, (int32_t)(n_items + e0), extra + 1, 0);
    } else {  // cannot be: see layout_max_popular
      atomicOr(status, kErrInput);
    }
  }
}

// The kHot items with the most entries of each minibatch (at least 2), most
// popular first, ties by id; -1 for unused slots.  Host side, at setup.
cudaError_t build_hot(const LayoutBuild& b, cudaStream_t st) {
  if (b.hot_item == nullptr) return cudaSuccess;
  const size_t FM = (size_t)b.F * (size_t)b.n_items;
  std::vector<int32_t> cnt(FM), hot((size_t)b.F * kHot, -1), idx((size_t)b.n_items);
  cudaError_t e = cudaMemcpyAsync(cnt.data(), b.item_cnt, sizeof(int32_t) * FM, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return e;
  for (int32_t mb = 0; mb < b.F; ++mb) {
    const int32_t* c = cnt.data() + (size_t)mb * b.n_items;
    for (int64_t j = 0; j < b.n_items; ++j) idx[j] = (int32_t)j;
    const int64_t h = std::min<int64_t>(kHot, b.n_items);
    std::partial_sort(idx.begin(), idx.begin() + h, idx.end(),
                      [c](int32_t x, int32_t y) { return c[x] != c[y] ? c[x] > c[y] : x < y; });
    for (int64_t r = 0; r < h && c[idx[r]] >= 2; ++r) hot[(size_t)mb * kHot + r] = idx[r];
  }
  e = cudaMemcpyAsync(b.hot_item, hot.data(), sizeof(int32_t) * hot.size(), cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e;
}

// A staged minibatch against the loaded one: every user id, item id and
// user offset must be equal; any difference latches kErrInput.
__global__ void stage_check_kernel(const int32_t* __restrict__ su, const int32_t* __restrict__ sj,
                                   const int32_t* __restrict__ suoff, const int32_t* __restrict__ ru,
                                   const int32_t* __restrict__ rj, const int32_t* __restrict__ ruoff, int64_t n,
                                   int64_t n_off, uint32_t* status) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n; k += stride)
    bad |= su[k] != ru[k] || sj[k] != rj[k];
  for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n_off; u += stride)
    bad |= suoff[u] != ruoff[u];
  if (__any_sync(0xffffffffu, bad) && (threadIdx.x & 31) == 0) atomicOr(status, kErrInput);
}

int blocks_for(int64_t n) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)sms * 16));
}

int64_t max_items(int64_t n_obs, int64_t n_users, int32_t F) {  // an item holds an entry or more
  return std::min(n_obs, layout_max_chunks(n_obs, F, n_users));
}

struct ScratchPlan {
  size_t val_out, cnt, nch, off, choff, hflag, hoff, hextra, ireps, cub, total;
  size_t cub_bytes;
};

ScratchPlan plan(int64_t n_obs, int64_t n_users, int64_t n_items, int32_t F) {
  ScratchPlan p{};
  const int64_t keys = (int64_t)F * n_users;
  size_t sort_bytes = 0, scan_bytes = 0, scan2_bytes = 0, scan3_bytes = 0;
  cub::DoubleBuffer<uint32_t> none(nullptr, nullptr);
  cub::DeviceRadixSort::SortPairs(nullptr, sort_bytes, none, none,
                                  (int)std::max<int64_t>(std::max(n_obs, n_users), 1), 0, 32);
  cub::DeviceScan::ExclusiveSum(nullptr, scan_bytes, (const int32_t*)nullptr, (int64_t*)nullptr, (int)(keys + 1));
  cub::DeviceScan::ExclusiveSum(nullptr, scan2_bytes, (const int32_t*)nullptr, (int32_t*)nullptr,
                                (int)(n_items + 1));
  scan_costs(nullptr, scan3_bytes, nullptr, max_items(n_obs, n_users, F), nullptr, nullptr);
  p.cub_bytes = std::max(std::max(sort_bytes, scan3_bytes), std::max(scan_bytes, scan2_bytes));
  size_t o = 0;
  auto take = [&o](size_t bytes) {
    const size_t at = o;
    o += align256(bytes);
    return at;
  };
  p.val_out = take(sizeof(uint32_t) * n_obs);
  p.cnt = take(sizeof(int32_t) * (keys + 1));
  p.nch = take(sizeof(int32_t) * (keys + 1));
  p.off = take(sizeof(int64_t) * (keys + 1));  // then the extra replica rows before each heavy user
  p.choff = take(sizeof(int64_t) * (keys + 1));
  p.hflag = take(sizeof(int32_t) * (keys + 1));
  p.hoff = take(sizeof(int64_t) * (keys + 1));
  p.hextra = take(sizeof(int32_t) * (keys + 1));
  p.ireps = take(sizeof(int32_t) * (n_items + 1));
  p.cub = take(p.cub_bytes);
  p.total = o;
  return p;
}

// The build's sorts in memory that the load has in hand for later: both buffers
// of the keys and one of the ids of n entries or items.
struct SortPlan {
  size_t key_in, key_out, val_in, total;
};
SortPlan sort_plan(int64_t n) {
  const size_t words = align256(sizeof(uint32_t) * (size_t)n);
  return SortPlan{0, words, 2 * words, 3 * words};
}

int bits_for(uint64_t max_key) {
  int b = 1;
  while (b < 32 && (max_key >> b) != 0) ++b;
  return b;
}

// Sorts n pairs on the keys' low bits, stable, between the two buffers of each
// (sorting into separate ones takes 8 bytes a pair more): ids in vals[0] on entry,
// sorted in *sorted, which is vals[0] or vals[1].
cudaError_t sort_ids(void* tmp, size_t bytes, uint32_t* key0, uint32_t* key1, uint32_t* val0, uint32_t* val1, int64_t n,
                     int bits, uint32_t** sorted, uint32_t** sorted_keys, cudaStream_t st) {
  cub::DoubleBuffer<uint32_t> keys(key0, key1), vals(val0, val1);
  const cudaError_t e = cub::DeviceRadixSort::SortPairs(tmp, bytes, keys, vals, (int)n, 0, bits, st);
  *sorted = vals.Current();
  *sorted_keys = keys.Current();
  return e;
}

}  // namespace

size_t layout_scratch_bytes(int64_t n_obs, int64_t n_users, int64_t n_items, int32_t F) {
  return plan(n_obs, n_users, n_items, F).total;
}

// In the stream's memory: the sort of the entries, then the work items in user
// order, then their summed costs.
size_t layout_stage_bytes(int64_t n_obs, int64_t n_users, int32_t F) {
  const int64_t items = max_items(n_obs, n_users, F);
  return std::max(sort_plan(n_obs).total, align256(std::max(sizeof(int4) * items, sizeof(int64_t) * (items + 1))));
}
// In the work list's: the sort of the items.
size_t layout_chunk_bytes(int64_t n_obs, int64_t n_users, int32_t F) {
  const int64_t items = max_items(n_obs, n_users, F);
  return std::max(sort_plan(items).total, sizeof(int4) * (size_t)layout_max_chunks(n_obs, F, n_users));
}

// A heavy segment has n > kHeavy >= kChunk entries and ceil(n/kChunk) < 2n/kChunk chunks.
// Every other user with entries in a minibatch adds one item.
int64_t layout_max_chunks(int64_t n_obs, int32_t F, int64_t n_users) {
  return 2 * n_obs / kChunk + F + 1 + std::min(n_obs, (int64_t)F * n_users);
}

// An item with extra replicas has more than kItemRep entries.
int64_t layout_max_popular(int64_t n_obs) { return n_obs / (kItemRep + 1) + 1; }

int64_t layout_max_heavy(int64_t n_obs, int32_t F) { return n_obs / (kHeavy + 1) + F + 1; }

// Replica rows: one per item plus the extra ones, sum (reps - 1) with reps - 1 < 3 mx / (2 kItemRep).
int64_t layout_max_item_reps(int64_t n_obs, int64_t n_items) { return n_items + 3 * n_obs / (2 * kItemRep) + 2; }

// Extra replica rows of heavy users: reps - 1 < 3 nch / (2 kUserRep), sum nch < 2 n_obs / kChunk.
int64_t layout_max_user_reps(int64_t n_obs) { return 3 * n_obs / (kChunk * kUserRep) + 2; }

cudaError_t build_layout(LayoutBuild& b, cudaStream_t st) {
  const ScratchPlan p = plan(b.n_obs, b.n_users, b.n_items, b.F);
  if (b.scratch_bytes < p.total) return cudaErrorInvalidValue;
  char* s = static_cast<char*>(b.scratch);
  const SortPlan q = sort_plan(b.n_obs);
  char* m = static_cast<char*>(b.stream_mem);
  uint32_t* key_in = reinterpret_cast<uint32_t*>(m + q.key_in);
  uint32_t* key_out = reinterpret_cast<uint32_t*>(m + q.key_out);
  uint32_t* val_in = reinterpret_cast<uint32_t*>(m + q.val_in);
  uint32_t* val_out = reinterpret_cast<uint32_t*>(s + p.val_out);
  int32_t* cnt = reinterpret_cast<int32_t*>(s + p.cnt);
  int64_t* off = reinterpret_cast<int64_t*>(s + p.off);
  int32_t* nch = reinterpret_cast<int32_t*>(s + p.nch);
  int64_t* choff = reinterpret_cast<int64_t*>(s + p.choff);
  int32_t* hflag = reinterpret_cast<int32_t*>(s + p.hflag);
  int64_t* hoff = reinterpret_cast<int64_t*>(s + p.hoff);
  int32_t* hextra = reinterpret_cast<int32_t*>(s + p.hextra);
  int64_t* hext = off;
  int32_t* ireps = reinterpret_cast<int32_t*>(s + p.ireps);
  void* cub_tmp = s + p.cub;
  const int64_t keys = (int64_t)b.F * b.n_users;
  uint32_t *perm = nullptr, *sorted = nullptr;
  cudaError_t e;

  for (void* z : {(void*)cnt, (void*)nch, (void*)hflag, (void*)hextra})
    if ((e = cudaMemsetAsync(z, 0, sizeof(int32_t) * (keys + 1), st)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(b.item_cnt, 0, sizeof(int32_t) * b.F * b.n_items, st)) != cudaSuccess) return e;
  keys_kernel<<<blocks_for(b.n_obs), 256, 0, st>>>(b.i, b.j, b.mb, b.n_obs, b.n_users, b.n_items, key_in, val_in, cnt,
                                                  b.item_cnt);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (b.n_obs > 0) {
    e = sort_ids(cub_tmp, p.cub_bytes, key_in, key_out, val_in, val_out, b.n_obs, bits_for((uint64_t)keys), &perm,
                 &sorted, st);
    if (e != cudaSuccess) return e;
    gather_kernel<<<blocks_for(b.n_obs), 256, 0, st>>>(perm, b.n_obs, b.i, b.j, b.D, b.rec_u, b.rec_j, b.rec_D);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  size_t tb = p.cub_bytes;
  if ((e = cub::DeviceScan::ExclusiveSum(cub_tmp, tb, cnt, off, (int)(keys + 1), st)) != cudaSuccess) return e;
  offsets_kernel<<<blocks_for((int64_t)b.F * (b.n_users + 1)), 256, 0, st>>>(off, b.n_users, b.F, b.uoff, b.mb_base,
                                                                            cnt, nch, hflag, hextra);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  tb = p.cub_bytes;
  if ((e = cub::DeviceScan::ExclusiveSum(cub_tmp, tb, nch, choff, (int)(keys + 1), st)) != cudaSuccess) return e;
  tb = p.cub_bytes;
  if ((e = cub::DeviceScan::ExclusiveSum(cub_tmp, tb, hflag, hoff, (int)(keys + 1), st)) != cudaSuccess) return e;
  tb = p.cub_bytes;
  if ((e = cub::DeviceScan::ExclusiveSum(cub_tmp, tb, hextra, hext, (int)(keys + 1), st)) != cudaSuccess) return e;
  item_reps_kernel<<<blocks_for(b.n_items + 1), 256, 0, st>>>(b.item_cnt, b.n_items, b.F, ireps);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  tb = p.cub_bytes;
  if ((e = cub::DeviceScan::ExclusiveSum(cub_tmp, tb, ireps, b.item_rep, (int)(b.n_items + 1), st)) != cudaSuccess)
    return e;
  popular_kernel<<<blocks_for(b.n_items), 256, 0, st>>>(b.item_rep, b.n_items, layout_max_popular(b.n_obs), b.popular,
                                                       b.n_popular, b.status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (b.n_obs > 0 && (e = build_hot(b, st)) != cudaSuccess) return e;
  // The work list, then its order: by tile of users and length, ties in user
  // order (the sort is stable).  The sort buffers of the entries are free now.
  int4* raw = static_cast<int4*>(b.stream_mem);
  int64_t* pre = static_cast<int64_t*>(b.stream_mem);
  const SortPlan qi = sort_plan(max_items(b.n_obs, b.n_users, b.F));
  key_in = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(b.chunk) + qi.key_in);
  key_out = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(b.chunk) + qi.key_out);
  val_in = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(b.chunk) + qi.val_in);
  const int64_t n_tiles = (b.n_users >> kTileBits) + 1;
  heavy_kernel<<<blocks_for(keys + 1), 256, 0, st>>>(
      choff, nch, hoff, hext, b.uoff, b.worker, b.n_users, b.F, raw, key_in, val_in, n_tiles, b.chunk_base,
      std::min(b.n_obs, b.max_chunks), b.heavy, b.heavy_base, b.max_heavy, layout_max_user_reps(b.n_obs), b.longest,
      b.status);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  int64_t n = 0;
  if ((e = cudaMemcpyAsync(&n, choff + keys, sizeof n, cudaMemcpyDeviceToHost, st)) != cudaSuccess) return e;
  if ((e = cudaStreamSynchronize(st)) != cudaSuccess) return e;
  if (n > std::min(b.n_obs, b.max_chunks)) return cudaErrorInvalidValue;
  b.pre = pre;
  b.n_work = n;
  // Users by worker (cnt, nch and hflag, [F n_users + 1] each, are free now).
  uint32_t* ids = reinterpret_cast<uint32_t*>(cnt);
  uint32_t* worker = reinterpret_cast<uint32_t*>(hflag);
  uint32_t* wuser = reinterpret_cast<uint32_t*>(b.wuser);
  iota_kernel<<<blocks_for(b.n_users), 256, 0, st>>>(ids, b.n_users);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  e = cudaMemcpyAsync(worker, b.worker, sizeof(int32_t) * b.n_users, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  e = sort_ids(cub_tmp, p.cub_bytes, worker, reinterpret_cast<uint32_t*>(nch), ids, wuser, b.n_users, bits_for(b.P), &perm,
               &sorted, st);
  if (e == cudaSuccess && perm != wuser)
    e = cudaMemcpyAsync(wuser, perm, sizeof(uint32_t) * b.n_users, cudaMemcpyDeviceToDevice, st);
  if (e != cudaSuccess) return e;
  worker_bases_kernel<<<b.P / 256 + 1, 256, 0, st>>>(sorted, b.n_users, b.P, b.wbase);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  if (n > 0) {
    e = sort_ids(cub_tmp, p.cub_bytes, key_in, key_out, val_in, val_out, n, bits_for((uint64_t)b.F * n_tiles << 7), &perm,
                 &sorted, st);
    // (the work list is written where the other buffers are)
    if (e == cudaSuccess && perm != val_out)
      e = cudaMemcpyAsync(val_out, perm, sizeof(uint32_t) * n, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return e;
  }
  place_items_kernel<<<blocks_for(n), 256, 0, st>>>(raw, val_out, n, b.chunk);
  if ((e = cudaGetLastError()) != cudaSuccess) return e;
  tb = p.cub_bytes;
  return scan_costs(cub_tmp, tb, b.chunk, n, pre, st);
}

// A round takes gpw * per_step places per step of its longest item, and the
// warps take whole rounds: those of a minibatch are its items gpw at a time, the
// last one partial.  With each item's entries rounded up to whole steps, a round's
// empty places are at most (gpw - 1) times the rise and fall of the lengths in it.
// Over a minibatch the lengths rise only from one tile of users to the next, so
// rise and fall add up to less than 2 kHeavy per tile, and to less than twice the
// entries.  A warp's first step is aligned.
int64_t layout_max_places(int64_t n_obs, int64_t n_users, int32_t F, const StreamGeometry& g, int64_t max_warps) {
  const int64_t items = max_items(n_obs, n_users, F);
  const int64_t warps = std::min((int64_t)F * max_warps, items / g.gpw + F);
  const int64_t tiles = (int64_t)F * ((n_users >> kTileBits) + 1), step = (int64_t)g.gpw * g.per_step;
  const int64_t uneven = std::min(2 * kHeavy * tiles, 2 * (n_obs + items * (g.per_step - 1)));
  const int64_t places = n_obs + items * (g.per_step - 1) + (g.gpw - 1) * uneven + F * g.gpw * (kHeavy + g.per_step);
  return std::min(step * n_obs, places) + kStepAlign * step * (warps + F);
}

cudaError_t launch_stage_check(const int32_t* su, const int32_t* sj, const int32_t* suoff, const int32_t* ru,
                               const int32_t* rj, const int32_t* ruoff, int64_t n, int64_t n_off, uint32_t* status,
                               cudaStream_t st) {
  stage_check_kernel<<<blocks_for(std::max(n, n_off)), 256, 0, st>>>(su, sj, suoff, ru, rj, ruoff, n, n_off, status);
  return cudaGetLastError();
}

cudaError_t launch_validate(const LayoutBuild& b, cudaStream_t st) {
  validate_kernel<<<blocks_for(std::max(b.n_obs, b.n_users)), 256, 0, st>>>(b.i, b.j, b.mb, b.n_obs, b.worker,
                                                                           b.n_users, b.n_items, b.F, b.P, b.status);
  return cudaGetLastError();
}

}  // namespace esspt
