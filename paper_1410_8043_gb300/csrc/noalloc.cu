// Per-worker objective for callers that must not allocate device memory.
//
// Some callers cannot call cudaMalloc (or any allocator): code that runs while
// a memory pool owned by someone else is the only source of device memory, a
// monitoring hook invoked from inside an application's hot loop where an
// allocation would synchronise the device or fragment the pool, or an
// embedded deployment with a fixed, pre-sized memory budget.  For them this
// file provides esspt_mf_worker_objective_noalloc(): the same per-entry
// objective as esspt_mf_objective(), summed per worker, whose accumulators
// live in a fixed array compiled into the library instead of in memory the
// caller hands over.
//
// Limits and behaviour:
//  - at most kNoAllocMaxWorkers workers (a 32 KB array, held by every GPU
//    that loads the library until the process exits); larger worker counts
//    are rejected with ESSPT_EINVAL before any work is queued;
//  - the first call on a device looks up the array's device address with the
//    device current (cudaGetSymbolAddress); make that first call outside any
//    stream capture;
//  - all calls share the one array and each call clears it first, so two
//    calls whose work overlaps on the GPU (different streams, no ordering
//    between them) race and may return mixed sums.
#include <mutex>

#include "internal.h"

namespace esspt {
namespace {

constexpr int32_t kNoAllocMaxWorkers = 2048;
constexpr int kMaxDevices = 64;

// Two fp64 sums per worker: sum e^2 at [p] and sum [e^2 + lambda(|L_i|^2+|R_j|^2)]
// at [kNoAllocMaxWorkers + p].
static __device__ __align__(256) double g_worker_sums[2 * kNoAllocMaxWorkers];

std::mutex g_mu;
double* g_sums_ptr[kMaxDevices] = {};

}  // namespace
}  // namespace esspt

extern "C" esspt_status esspt_mf_worker_objective_noalloc(esspt_ctx* ctx, int32_t version, float lambda,
                                                          double* h_sq, double* h_pen) {
  using namespace esspt;
  if (!ctx) return ESSPT_EINVAL;
  ObjectiveArgs a;
  cudaStream_t st = nullptr;
  const esspt_status s = mf_view(ctx, version, &a, &st);
  if (s != ESSPT_OK) return s;
  const int32_t P = a.P;
  if (!h_sq || !h_pen) return mf_fail(ctx, ESSPT_EINVAL, "null output");
  if (P > kNoAllocMaxWorkers)
    return mf_fail(ctx, ESSPT_EINVAL,
                               "esspt_mf_worker_objective_noalloc: more than 2048 workers do not fit its fixed "
                               "accumulator array; use esspt_mf_objective");
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return mf_fail(ctx, ESSPT_ECUDA, cudaGetErrorString(e));
  if (dev < 0 || dev >= kMaxDevices) return mf_fail(ctx, ESSPT_EINVAL, "device ordinal too large");
  double* sums = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_mu);
    if (!g_sums_ptr[dev]) {
      void* p = nullptr;
      e = cudaGetSymbolAddress(&p, g_worker_sums);
      if (e != cudaSuccess) return mf_fail(ctx, ESSPT_ECUDA, cudaGetErrorString(e));
      g_sums_ptr[dev] = static_cast<double*>(p);
    }
    sums = g_sums_ptr[dev];
  }
  // Every call starts from zero: the array keeps the previous call's sums.
  e = cudaMemsetAsync(sums, 0, sizeof(double) * 2 * kNoAllocMaxWorkers, st);
  a.lambda = lambda;
  a.out = sums;
  a.out_stride = kNoAllocMaxWorkers;
  if (e == cudaSuccess) e = launch_worker_objective(a, st);
  if (e == cudaSuccess) e = cudaMemcpyAsync(h_sq, sums, sizeof(double) * P, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(h_pen, sums + kNoAllocMaxWorkers, sizeof(double) * P, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return mf_fail(ctx, ESSPT_ECUDA, cudaGetErrorString(e));
  return ESSPT_OK;
}
