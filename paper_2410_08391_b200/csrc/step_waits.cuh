// Bounded waits of the persistent step kernels (step_mega_mma.cu, step_mega.cu): tagged values in global memory, and the waits of the
// former's loader warps.  In a header of their own so that the self-test of selftest.cu runs the same code.
#pragma once
#include "common.cuh"
#include "tc_ptx.cuh"

namespace tcp {

constexpr unsigned LAZY_LIMIT = 10u * 1000u * 1000u;         // polls with a sleep between them: 0.2 us each (measured), two seconds

typedef unsigned long long u64;

// Wait on an mbarrier: the test of a phase that is complete already costs 20 cycles, the bounded loop is kept out of line.
__device__ __forceinline__ bool slow_wait(uint32_t bar, uint32_t parity, volatile int* s_abort, int* status) {
  return !*s_abort && mbar_wait(bar, parity, s_abort, status);
}
__device__ __forceinline__ bool quick_wait(uint32_t bar, uint32_t parity, volatile int* s_abort, int* status) {
  return mbar_test(bar, parity) || slow_wait(bar, parity, s_abort, status);
}

// Wait of a loader warp, which is far ahead of its consumers: one lane looks now and then, so that the wait takes neither
// issue slots nor shared-memory cycles from them.  (A consumer that has given up releases no slot: the copy into it
// may still be in flight, and the loader would arm its barrier a second time.)
__device__ __forceinline__ bool lazy_wait(uint32_t bar, uint32_t parity, volatile int* s_abort, int* status, unsigned limit = LAZY_LIMIT) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) {
    unsigned it = 0;
    while (!mbar_poll(bar, parity)) {
      if (*s_abort) { ok = 0; break; }
      if (++it > limit) { *s_abort = 1; dev_flag(status, DEV_TIMEOUT); ok = 0; break; }
      __nanosleep(100);
    }
  }
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// Tagged values: the value's bits in the low word, the tag in the high word, always stored and loaded as one 64-bit word.
__device__ __forceinline__ void ll_store(u64* p, float v, uint32_t tag) {
  asm volatile("st.relaxed.gpu.global.b64 [%0], %1;" ::"l"(p), "l"((u64)tag << 32 | __float_as_uint(v)) : "memory");
}
__device__ __forceinline__ u64 ll_load(const u64* p) {
  u64 v;
  asm volatile("ld.relaxed.gpu.global.b64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void ll_load2(const u64* p, u64& a, u64& b) {
  asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p) : "memory");
}
__device__ __forceinline__ float ll_val(u64 v) { return __uint_as_float((uint32_t)v); }
__device__ __forceinline__ uint32_t ll_tag(u64 v) { return (uint32_t)(v >> 32); }
// One poll more; false = the wait is over without its value (ran out, or another role gave up).
__device__ __forceinline__ bool poll_more(unsigned& it, volatile int* s_abort, int* status, unsigned limit = L2_POLL_LIMIT) {
  ++it;
  if ((it & 63u) == 0u) {
    if (*s_abort) return false;
    if (*reinterpret_cast<volatile int*>(status) == DEV_TIMEOUT) { *s_abort = 1; return false; }
  }
  if (it > limit) { *s_abort = 1; dev_flag(status, DEV_TIMEOUT); return false; }
  return true;
}
// A value of the wanted tag.
__device__ __forceinline__ float ll_wait(const u64* p, uint32_t tag, bool& dead, volatile int* s_abort, int* status,
                                         unsigned limit = L2_POLL_LIMIT) {
  u64 v = ll_load(p);
  unsigned it = 0;
  while (ll_tag(v) != tag && !dead) {
    if (!poll_more(it, s_abort, status, limit)) dead = true;
    v = ll_load(p);
  }
  return ll_val(v);
}

}  // namespace tcp
