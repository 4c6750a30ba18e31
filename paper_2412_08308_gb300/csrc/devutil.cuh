// Small sm_103a device helpers: mbarriers, 1-D bulk TMA copies, cp.async and
// bounded waits.  Every wait in this library gives up after a clock budget and
// reports failure instead of spinning forever.
#pragma once

#include <cstdint>

namespace swgb {

// ~1 s at GB300 clocks: a wait that has not completed by then is reported as
// a timeout (status SW_ETIMEOUT) and the kernel returns.
constexpr long long kWaitBudgetCycles = 2000000000LL;

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// Wait for the phase with the given parity to complete; false on timeout.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > kWaitBudgetCycles) return false;
  }
  return true;
}

// 1-D bulk copy global -> shared through the TMA unit, completing on `bar`.
// dst, src and bytes must be multiples of 16.
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Per-thread asynchronous 16-byte copy global -> shared (L2 only).
__device__ __forceinline__ void cp_async16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Release/acquire flags between CTAs (gpu scope).
__device__ __forceinline__ int32_t ld_acquire(const int32_t *p) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

__device__ __forceinline__ void st_release(int32_t *p, int32_t v) {
  asm volatile("st.release.gpu.global.s32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Relaxed 64-bit accesses at gpu scope: single-copy atomic, served by L2 (never
// a stale L1 line), no ordering against other accesses.
__device__ __forceinline__ unsigned long long ld_relaxed_u64(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p));
  return v;
}

__device__ __forceinline__ void st_relaxed_u64(unsigned long long *p, unsigned long long v) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v));
}

// Two 64-bit words by one 128-bit store (p 16-byte aligned), each word
// single-copy atomic like st_relaxed_u64, with no order between them.
__device__ __forceinline__ void st_relaxed_2xu64(unsigned long long *p, uint32_t lo0, uint32_t hi0, uint32_t lo1,
                                                 uint32_t hi1) {
  const unsigned long long v0 = ((unsigned long long)hi0 << 32) | lo0, v1 = ((unsigned long long)hi1 << 32) | lo1;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(v0), "l"(v1));
}

// A wait on another warp of a long pipeline, which may legitimately last as
// long as a whole band takes: ~60 s at GB300 clocks.
constexpr long long kLongWaitBudgetCycles = 120000000000LL;

// Wait until *p >= v (published by another CTA or warp) and return the value
// read; a value < v means the clock budget ran out.
__device__ __forceinline__ int32_t wait_flag_value(const int32_t *p, int32_t v, long long budget) {
  int32_t cur = ld_acquire(p);
  if (cur >= v) return cur;
  const long long t0 = clock64();
  while ((cur = ld_acquire(p)) < v) {
    if (clock64() - t0 > budget) return cur;
    __nanosleep(128);
  }
  return cur;
}

}  // namespace swgb
