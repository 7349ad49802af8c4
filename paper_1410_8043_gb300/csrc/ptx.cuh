// Small inline-PTX helpers: vector loads/stores with L2 eviction hints, packed
// fp32 arithmetic, and vector fp32 reductions into global memory.
#pragma once

#include <stdint.h>

namespace esspt {

__device__ __forceinline__ uint64_t policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Predicated forms: the access happens only when `pred` is true, without a
// branch around the asm (loads give zeros when it is false).
__device__ __forceinline__ float4 ld_stream_if(const float4* p, uint64_t pol, bool pred) {
  float4 r;
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n mov.f32 %0, 0f00000000;\n mov.f32 %1, 0f00000000;\n"
      " mov.f32 %2, 0f00000000;\n mov.f32 %3, 0f00000000;\n"
      " @q ld.global.L1::no_allocate.L2::cache_hint.v4.f32 {%0,%1,%2,%3}, [%4], %6;\n}"
      : "=f"(r.x), "=f"(r.y), "=f"(r.z), "=f"(r.w)
      : "l"(p), "r"((int)pred), "l"(pol));
  return r;
}

__device__ __forceinline__ void st_stream_if(float4* p, float4 v, uint64_t pol, bool pred) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n"
      " @q st.global.L1::no_allocate.L2::cache_hint.v4.f32 [%0], {%1,%2,%3,%4}, %6;\n}"
      :
      : "l"(p), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w), "r"((int)pred), "l"(pol)
      : "memory");
}

// 16-byte asynchronous global -> shared copies, bypassing L1 with an L2
// eviction-priority policy for the source lines, and through L1; nothing
// happens when `pred` is false.
__device__ __forceinline__ void cp_async16_hint_if(void* smem, const void* gmem, bool pred, uint64_t pol) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n"
      " @q cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %3;\n}" ::"r"(s),
      "l"(gmem), "r"((int)pred), "l"(pol)
      : "memory");
}
__device__ __forceinline__ void cp_async16_if(void* smem, const void* gmem, bool pred) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %2, 0;\n @q cp.async.ca.shared.global [%0], [%1], 16;\n}" ::"r"(s),
               "l"(gmem), "r"((int)pred)
               : "memory");
}
// Streaming 32-bit load (read once per clock): skip L1, evict-first in L2.
__device__ __forceinline__ int32_t ld_stream_i32(const int32_t* p, uint64_t pol) {
  int32_t r;
  asm volatile("ld.global.L1::no_allocate.L2::cache_hint.b32 %0, [%1], %2;" : "=r"(r) : "l"(p), "l"(pol));
  return r;
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// Wait for all of the thread's asynchronous copies, or until at most N of its
// newest groups are in flight.
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// out[0..3] += v, performed at L2 (no return value).
__device__ __forceinline__ void red_add_v4(float4* p, float4 v) { atomicAdd(p, v); }

// One float4 slice as two packed fp32 pairs, the operands of the packed fp32
// instructions (sm_100 and later): two IEEE fp32 operations per instruction,
// each rounded as its scalar form.
typedef unsigned long long u64;
struct f2x2 {
  u64 lo, hi;
};
__device__ __forceinline__ u64 pack2(float x, float y) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
  return r;
}
__device__ __forceinline__ void unpack2(u64 v, float& x, float& y) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(x), "=f"(y) : "l"(v));
}
__device__ __forceinline__ float sum2(u64 v) {
  float x, y;
  unpack2(v, x, y);
  return x + y;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// r = *p when `pred`, else r as it was; through L1.  The second form (.nc) is
// for memory that no kernel writes while the reading one is resident: not for
// ring rows in a kernel that may start beside the clock before it
// (await_previous_kernel orders ordinary accesses only).
__device__ __forceinline__ void ld_f2x2_if(f2x2& r, const float4* p, bool pred) {
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %3, 0;\n @q ld.global.v2.b64 {%0, %1}, [%2];\n}"
               : "+l"(r.lo), "+l"(r.hi)
               : "l"(p), "r"((int)pred));
}
__device__ __forceinline__ void ldg_f2x2_if(f2x2& r, const float4* p, bool pred) {
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %3, 0;\n @q ld.global.nc.v2.b64 {%0, %1}, [%2];\n}"
               : "+l"(r.lo), "+l"(r.hi)
               : "l"(p), "r"((int)pred));
}
__device__ __forceinline__ f2x2 lds_f2x2(const float4* p) {
  const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(p);
  return f2x2{v.x, v.y};
}
__device__ __forceinline__ void st_f2x2(float4* p, u64 lo, u64 hi) {
  *reinterpret_cast<ulonglong2*>(p) = make_ulonglong2(lo, hi);
}
__device__ __forceinline__ void st_stream_f2x2_if(float4* p, u64 lo, u64 hi, uint64_t pol, bool pred) {
  asm volatile(
      "{\n .reg .pred q;\n setp.ne.b32 q, %4, 0;\n"
      " @q st.global.L1::no_allocate.L2::cache_hint.v2.b64 [%0], {%1, %2}, %3;\n}" ::"l"(p),
      "l"(lo), "l"(hi), "l"(pol), "r"((int)pred)
      : "memory");
}
// p[0..3] += (lo, hi) when `pred`, performed at L2 (vector reduction, sm_90
// and later), predicated inside the asm so that no branch surrounds it.
__device__ __forceinline__ void red_add_f2x2_if(float4* p, u64 lo, u64 hi, bool pred) {
  float a, b, c, d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(lo));
  asm("mov.b64 {%0, %1}, %2;" : "=f"(c), "=f"(d) : "l"(hi));
  asm volatile("{\n .reg .pred q;\n setp.ne.b32 q, %5, 0;\n @q red.global.add.v4.f32 [%0], {%1,%2,%3,%4};\n}" ::"l"(p),
               "f"(a), "f"(b), "f"(c), "f"(d), "r"((int)pred)
               : "memory");
}

// Programmatic dependent launch: a kernel launched with it may start while the
// kernel before it in the stream still runs; it waits here, before its first
// access to global memory, until that one (and so all before it) has finished
// and its writes are visible to ordinary accesses.  Memory that a kernel may
// write is therefore read with ordinary loads here, never as read-only data
// (.nc, __ldg, const __restrict__), which must not change while the reading
// kernel is resident.  Then it lets the next such kernel start.
__device__ __forceinline__ void await_previous_kernel() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// SplitMix64 (Steele, Lea and Flood, OOPSLA 2014): output n of the sequence
// whose state starts at s0 is mix64(s0 + n * 0x9E3779B97F4A7C15).
__host__ __device__ __forceinline__ uint64_t mix64(uint64_t z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Draw `index` of stream `stream` under `seed`: output index+1 of SplitMix64
// started at state mix64(seed) ^ mix64(stream).
__host__ __device__ __forceinline__ uint64_t ctr_u64(uint64_t seed, uint64_t stream, uint64_t index) {
  const uint64_t s0 = mix64(seed) ^ mix64(stream);
  return mix64(s0 + (index + 1ull) * 0x9E3779B97F4A7C15ull);
}

}  // namespace esspt
