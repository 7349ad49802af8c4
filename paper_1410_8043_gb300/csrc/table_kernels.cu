// Table kernels: the read-version schedule, the Clock() copy-forward of the
// version ring, and the generic GET / INC row kernels.
#include <algorithm>
#include <cmath>

#include "chained.cuh"
#include "internal.h"
#include "ptx.cuh"
#include "schedule.cuh"

namespace esspt {

// ---------------------------------------------------------------------------
// Schedule: v_p(c) for every worker p; one thread per worker (the rule is in
// schedule.cuh).  The MF clock computes the next schedule inside its item
// merge kernel instead of launching this one.
// ---------------------------------------------------------------------------
__global__ void schedule_kernel(ScheduleArgs a) {
  await_previous_kernel();
  for (int32_t p = blockIdx.x * blockDim.x + threadIdx.x; p < a.P; p += gridDim.x * blockDim.x)
    schedule_worker(a, p);
}

cudaError_t launch_schedule(const ScheduleArgs& a, cudaStream_t st) {
  const int threads = 256;
  const int blocks = (int)std::min<int64_t>((a.P + threads - 1) / threads, 1024);
  return launch_chained(schedule_kernel, blocks, threads, st, true, a);
}

// ---------------------------------------------------------------------------
// VAP in-transit norms (Sec. 2.1): for k = 1..kmax, the max over the table of
// |X[c-1] - X[c-1-k]|, folded per block and combined with an integer atomic
// max on the bits of the non-negative fp32 value (which orders like the
// value).  Candidates are taken 8 at a time so that each pass reads X[c-1]
// once for 8 older versions.
// ---------------------------------------------------------------------------
constexpr int kVapBatch = 8;  // candidates per launch

__device__ __forceinline__ float vap_absdiff_max(float m, float4 a, float4 b) {
  const float d0 = fabsf(a.x - b.x), d1 = fabsf(a.y - b.y), d2 = fabsf(a.z - b.z), d3 = fabsf(a.w - b.w);
  // fmaxf drops NaN; a NaN difference must fail the bound, so it becomes +inf.
  const bool nan = (d0 != d0) || (d1 != d1) || (d2 != d2) || (d3 != d3);
  return nan ? __int_as_float(0x7f800000) : fmaxf(fmaxf(m, fmaxf(d0, d1)), fmaxf(d2, d3));
}

__global__ void __launch_bounds__(256) vap_norms_kernel(const float4* __restrict__ ring, int64_t slot4, int32_t nslots,
                                                        int32_t c, int32_t k0, int32_t nk, uint32_t* __restrict__ norm) {
  __shared__ float red[kVapBatch][8];
  float m[kVapBatch];
#pragma unroll
  for (int t = 0; t < kVapBatch; ++t) m[t] = 0.f;
  const float4* cur = ring + (int64_t)((c - 1) % nslots) * slot4;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < slot4; q += stride) {
    const float4 x = cur[q];
#pragma unroll
    for (int t = 0; t < kVapBatch; ++t) {
      if (t < nk) {
        const int32_t ver = c - 1 - (k0 + t);
        m[t] = vap_absdiff_max(m[t], x, ring[(int64_t)(ver % nslots) * slot4 + q]);
      }
    }
  }
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
  for (int t = 0; t < kVapBatch; ++t) {
    float v = m[t];
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, off));
    if (lane == 0) red[t][wid] = v;
  }
  __syncthreads();
  if (threadIdx.x < kVapBatch && (int)threadIdx.x < nk) {
    float v = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) v = fmaxf(v, red[threadIdx.x][w]);
    if (v > 0.f) atomicMax(norm + k0 + threadIdx.x, __float_as_uint(v));
  }
}

// ---------------------------------------------------------------------------
// The same on large tables: which of the versions c-1-k, k = k0 .. k1, have an
// in-transit max-norm |X[c-1] - X[c-1-k]| (over the table, fp32) within the
// bound; norm[k] stays 0 if so and becomes +inf if not.  Only the stalest one within the bound
// is read, so the candidates are taken from the stalest down, each until an
// element breaks the bound, and none after one has been scanned whole: two
// tables are read where all candidates at once would take k1 + 1 of them (s = 3
// on a 498k x 100 table: 160 us with each norm taken in full).
//
// The work is one sequence of pieces, candidate by candidate, that the blocks
// draw from a ticket (words[0]); a broken bound moves the ticket on to the next
// candidate.  A block never waits: while a candidate's last pieces are with
// other blocks it takes pieces of the next one, which may turn out needless.
// words[k] counts the scanned pieces of candidate k.
// ---------------------------------------------------------------------------
constexpr int kVapLoads = 8;  // float4 of each version per thread and piece
constexpr int64_t kVapPiece = 256 * kVapLoads;

// A NaN difference counts as +inf.
__device__ __forceinline__ bool vap_breaks(float4 a, float4 b, float bound) {
  const float d0 = fabsf(a.x - b.x), d1 = fabsf(a.y - b.y), d2 = fabsf(a.z - b.z), d3 = fabsf(a.w - b.w);
  const float m = fmaxf(fmaxf(d0, d1), fmaxf(d2, d3));  // drops NaN
  const bool nan = (d0 != d0) || (d1 != d1) || (d2 != d2) || (d3 != d3);
  return m > bound || (nan && bound < __int_as_float(0x7f800000));
}

__global__ void __launch_bounds__(256) vap_scan_kernel(const float4* __restrict__ ring, int64_t slot4, int32_t nslots,
                                                       int32_t c, int32_t k0, int32_t k1, int32_t kmax, float bound,
                                                       uint32_t pieces, uint32_t* norm, uint32_t* words) {
  __shared__ uint32_t ticket;
  volatile uint32_t* vnorm = norm;
  volatile uint32_t* vwords = words;
  if (k1 < kmax && vnorm[k1 + 1] == 0u) return;  // an earlier launch found the version
  const uint32_t last = (uint32_t)(k1 - k0 + 1) * pieces;
  const float4* cur = ring + (int64_t)((c - 1) % nslots) * slot4;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t t = atomicAdd(words, 1u);
      // A candidate before this one that is scanned whole within its bound ends the search.
      if (t < last)
        for (int32_t k = k1; k > k1 - (int32_t)(t / pieces); --k)
          if (vnorm[k] == 0u && vwords[k] == pieces) t = last;
      ticket = t;
    }
    __syncthreads();
    const uint32_t t = ticket;
    if (t >= last) return;
    const int32_t k = k1 - (int32_t)(t / pieces);
    const float4* old = ring + (int64_t)((c - 1 - k) % nslots) * slot4;
    const uint32_t p = t % pieces;  // taken from both ends in turn
    const int64_t q0 = (int64_t)((p & 1u) ? pieces - 1u - p / 2u : p / 2u) * kVapPiece + threadIdx.x;
    bool breaks = false;
    float4 x[kVapLoads], y[kVapLoads];
#pragma unroll
    for (int i = 0; i < kVapLoads; ++i) {
      const int64_t q = min(q0 + 256 * i, slot4 - 1);
      x[i] = cur[q];
      y[i] = old[q];
    }
#pragma unroll
    for (int i = 0; i < kVapLoads; ++i) breaks |= vap_breaks(x[i], y[i], bound);
    breaks = __syncthreads_or(breaks);
    if (threadIdx.x == 0) {
      if (breaks) {
        vnorm[k] = 0x7f800000u;
        atomicMax(words, (t / pieces + 1u) * pieces);
      } else {
        __threadfence();
        atomicAdd(words + k, 1u);
      }
    }
  }
}

cudaError_t launch_vap(const float* ring, int64_t slot_floats, int32_t nslots, int32_t c, int32_t kmax,
                            double bound, uint32_t* norm, uint32_t* words, cudaStream_t st) {
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // The largest fp32 value within the bound: fp32 norms compare with it as with the bound.
  float fb = (float)bound;
  if ((double)fb > bound) fb = std::nextafterf(fb, 0.f);
  const int64_t slot4 = slot_floats / 4, pieces = (slot4 + kVapPiece - 1) / kVapPiece;
  // The scan saves up to kmax - 1 tables of traffic and costs its tickets, about
  // 10 us (4 MB table, kmax = 6: 17 us against 7 for all norms at once).  Its worst
  // case is one element, far from both ends of the table, that breaks every
  // candidate: each is read nearly whole, 2 kmax tables where the norms read kmax +
  // 1 (the newest version's from L2).  48 MB table, whole CLOCK, norms against scan:
  // kmax = 4: 67 us, 40 with the stalest version in bound, 47 broken at an end of
  // the table, 62 in its middle; kmax = 8: 112, 41, 92, 127.
  if ((kmax - 1) * slot_floats * 4 < (128 << 20)) {
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((slot4 + 255) / 256, (int64_t)sms * 8));
    for (int32_t k0 = 1; k0 <= kmax; k0 += kVapBatch) {
      vap_norms_kernel<<<blocks, 256, 0, st>>>(reinterpret_cast<const float4*>(ring), slot4, nslots, c, k0,
                                               std::min(kVapBatch, kmax - k0 + 1), norm);
      const cudaError_t e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
  }
  for (int32_t k1 = kmax; k1 >= 1; k1 -= kVapBatch) {
    const int32_t k0 = std::max(1, k1 - kVapBatch + 1);
    if (k1 < kmax) {
      const cudaError_t e = cudaMemsetAsync(words, 0, sizeof(uint32_t), st);
      if (e != cudaSuccess) return e;
    }
    const int blocks = (int)std::min<int64_t>(pieces * (k1 - k0 + 1), (int64_t)sms * 8);
    vap_scan_kernel<<<blocks, 256, 0, st>>>(reinterpret_cast<const float4*>(ring), slot4, nslots, c, k0, k1, kmax, fb,
                                            (uint32_t)pieces, norm, words);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Copy-forward: slot(c) <- slot(c-1) for a range of rows, so that the
// deltas of clock c can land in place (Clock() merge, Sec. 2.1 / Sec. 4).
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) copy_rows_kernel(float4* dst, const float4* src, int64_t n4) {
  await_previous_kernel();
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (; k + 3 * stride < n4; k += 4 * stride) {
    const float4 a = src[k], b = src[k + stride], c = src[k + 2 * stride], d = src[k + 3 * stride];
    dst[k] = a;
    dst[k + stride] = b;
    dst[k + 2 * stride] = c;
    dst[k + 3 * stride] = d;
  }
  for (; k < n4; k += stride) dst[k] = src[k];
}

cudaError_t launch_copy_rows(float* dst, const float* src, int64_t n_floats, cudaStream_t st) {
  const int64_t n4 = n_floats / 4;
  if (n4 == 0) return cudaSuccess;
  int dev = 0, sms = 148;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int threads = 256;
  const int64_t want = (n4 + threads * 4 - 1) / (threads * 4);
  const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)sms * 8));
  return launch_chained(copy_rows_kernel, blocks, threads, st, true, reinterpret_cast<float4*>(dst),
                        reinterpret_cast<const float4*>(src), n4);
}

// ---------------------------------------------------------------------------
// GET: rows of worker p's read version; INC: additive updates into the version
// being written (Sec. 2.1, Sec. 4).  A program calls these for each worker in
// turn, a few thousand rows at a time, so a call's length is its launch and one
// chain of loads: lanes of a power of two of at least K/4 (32 at most) take a
// row, the row groups of a warp as many rows, and a call starts while the kernel
// before it drains.  One warp per row and ordinary launches: 4.2 and 3.8 us for
// 2001 rows of 64 values.
// ---------------------------------------------------------------------------
struct RowLanes {  // the row group of a thread
  int64_t first, stride;
  int lane, lanes;
  __device__ explicit RowLanes(int log_lanes)
      : first(((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> log_lanes),
        stride(((int64_t)gridDim.x * blockDim.x) >> log_lanes),
        lane(threadIdx.x & ((1 << log_lanes) - 1)),
        lanes(1 << log_lanes) {}
};

__global__ void __launch_bounds__(256) get_rows_kernel(const float* ring, int64_t n_rows, int32_t K, int32_t nslots,
                                                       const int32_t* v, int32_t worker, const int32_t* ids, int64_t n,
                                                       float* out, uint32_t* status, int32_t* rowver, int32_t c,
                                                       int32_t s, int32_t* vmin, int log_lanes) {
  await_previous_kernel();
  const RowLanes g(log_lanes);
  const int32_t K4 = K >> 2;
  const int32_t wslot = rowver ? 0 : v[worker] % nslots;
  int32_t oldest = 0x7fffffff;
  for (int64_t k = g.first; k < n; k += g.stride) {
    const int32_t r = ids[k];
    if (r < 0 || r >= n_rows) {
      if (g.lane == 0) atomicOr(status, kErrRowRange);
      continue;
    }
    int32_t slot = wslot;
    if (rowver) {
      // Row-granular cache: refresh the row to c-1 if it is missing or too
      // stale (every refresh of it in this clock writes the same value, so
      // lanes that read before and after one agree).
      int32_t* V = rowver + (int64_t)worker * n_rows + r;
      int32_t ver = *V;
      if (ver < 0 || ver < c - 1 - s) {
        ver = c - 1;
        if (g.lane == 0) *V = ver;
      }
      oldest = min(oldest, ver);
      slot = ver % nslots;
    }
    const float4* src = reinterpret_cast<const float4*>(ring) + ((int64_t)slot * n_rows + r) * K4;
    float4* o = reinterpret_cast<float4*>(out + k * K);
#pragma unroll 1
    for (int32_t q = g.lane; q < K4; q += g.lanes) o[q] = src[q];
  }
  if (vmin != nullptr) {
    oldest = __reduce_min_sync(0xffffffffu, oldest);
    if ((threadIdx.x & 31) == 0 && oldest != 0x7fffffff) atomicMin(vmin, oldest);
  }
}

__global__ void __launch_bounds__(256) inc_rows_kernel(float* slot, int64_t n_rows, int32_t K, const int32_t* ids,
                                                       const float* d, int64_t n, uint32_t* status, int log_lanes) {
  await_previous_kernel();
  const RowLanes g(log_lanes);
  const int32_t K4 = K >> 2;
  for (int64_t k = g.first; k < n; k += g.stride) {
    const int32_t r = ids[k];
    if (r < 0 || r >= n_rows) {
      if (g.lane == 0) atomicOr(status, kErrRowRange);
      continue;
    }
    float4* dst = reinterpret_cast<float4*>(slot) + (int64_t)r * K4;
    const float4* src = reinterpret_cast<const float4*>(d + k * K);
    for (int32_t q = g.lane; q < K4; q += g.lanes) red_add_v4(dst + q, src[q]);
  }
}

namespace {
int log_lanes_for(int32_t K) {
  int log = 0;
  while (log < 5 && (1 << log) < K / 4) ++log;
  return log;
}
int row_blocks(int64_t n, int log_lanes) { return (int)std::min<int64_t>(((n << log_lanes) + 255) / 256, 4096); }
}  // namespace

cudaError_t launch_get(const float* ring, int64_t n_rows, int32_t K, int32_t nslots, const int32_t* v, int32_t worker,
                       const int32_t* ids, int64_t n, float* out, uint32_t* status, int32_t* rowver, int32_t c,
                       int32_t s, int32_t* vmin, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int log = log_lanes_for(K);
  return launch_chained(get_rows_kernel, row_blocks(n, log), 256, st, true, ring, n_rows, K, nslots, v, worker, ids, n,
                        out, status, rowver, c, s, vmin, log);
}

cudaError_t launch_inc(float* slot, int64_t n_rows, int32_t K, const int32_t* ids, const float* d, int64_t n,
                       uint32_t* status, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const int log = log_lanes_for(K);
  return launch_chained(inc_rows_kernel, row_blocks(n, log), 256, st, true, slot, n_rows, K, ids, d, n, status, log);
}

}  // namespace esspt
