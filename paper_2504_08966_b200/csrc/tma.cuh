// mbarrier primitives of the kernels that stage data through shared memory with tiled bulk copies (TMA).
// Every wait is bounded: after kWaitNs of wall time it returns false and the caller gives up cleanly.
#pragma once
#include <stdint.h>

#include <cuda/annotated_ptr>

#include "../../include/pact.h"

namespace pact {

constexpr unsigned long long kWaitNs = 1000000000ull;   // one second per wait, then give up

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
  return ok != 0;
}
// The same, but the thread may sleep for up to 20 us in it: wakes later, takes no power meanwhile.
__device__ __forceinline__ bool mbar_try_wait_asleep(uint64_t *bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity), "r"(20000u) : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait: false when kWaitNs of wall time have passed without the phase completing.
static __device__ __noinline__ bool mbar_wait_slow(uint64_t *bar, uint32_t parity) {
  const unsigned long long t0 = global_ns();
  for (uint32_t i = 0;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 255u) == 255u && global_ns() - t0 > kWaitNs) return false;
  }
}
template <bool ASLEEP = false>
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity) {
  for (int i = 0; i < 64; ++i)
    if (ASLEEP ? mbar_try_wait_asleep(bar, parity) : mbar_try_wait(bar, parity)) return true;
  return mbar_wait_slow(bar, parity);
}

// Untiled bulk copy from global to this CTA's shared memory: addresses and size multiples of 16 bytes; the bytes are
// reported to `bar`.  One such copy occupies an SM's copy engine for about 28 ns or its size at 128 GB/s, whichever is
// longer, so rows of a few KB are what it is for: measured on one SM 120-134 GB/s from the L2 and 115 GB/s from HBM,
// against 109 and 45 GB/s with 16-byte loads to registers and 52 GB/s with 16-byte asynchronous copies.
__device__ __forceinline__ void bulk_load(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

// Loads that say what the L2 is to do with their lines.  The policies are the words of CUDA's access properties, known when the kernels are
// compiled; made by createpolicy in the kernels they would take two registers where the token pass already spills some.
constexpr uint64_t kEvictNormal = static_cast<uint64_t>(cuda::access_property(cuda::access_property::normal{}));
constexpr uint64_t kEvictFirst = static_cast<uint64_t>(cuda::access_property(cuda::access_property::streaming{}));   // (the first to be replaced)
__device__ __forceinline__ void bulk_load_hint(void *dst, const void *src, uint32_t bytes, uint64_t *bar, uint64_t policy) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1], %2, [%3], %4;"
               ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy) : "memory");
}
__device__ __forceinline__ uint4 ld_hint(const void *p, uint64_t policy) {   // of an input
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.L2::cache_hint.v4.u32 {%0, %1, %2, %3}, [%4], %5;" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p), "l"(policy));
  return v;
}

// The same way back, 16-byte aligned, a multiple of 16 bytes; after bulk_store_wait the shared memory of the thread's copies
// so far has been read, and the kernels after this one find the data.
__device__ __forceinline__ void bulk_store(void *dst, const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_u32(src)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_store_wait() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// For a CTA that gives up after a wait that ran out: the copies it has under way still write to its shared memory, which the
// next CTA may have by then.  Threads 0 .. n - 1 wait for a barrier each, whichever its phase: the wait for the phase that is
// over returns at once, and one for which nothing was asked runs out.  (A call, out of the way of the code that runs.)
static __device__ __noinline__ void land_copies(uint64_t *bars, int n) {
  if ((int)threadIdx.x < n) {
    mbar_wait_slow(bars + threadIdx.x, 0);
    mbar_wait_slow(bars + threadIdx.x, 1);
  }
}

// Wait of a whole warp: one lane polls (32 lanes spinning on one barrier word get in the way of the
// copy engine that has to update it), the result is shared.
template <bool ASLEEP = false>
__device__ __forceinline__ bool mbar_wait_warp(uint64_t *bar, uint32_t parity) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait<ASLEEP>(bar, parity) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

// The same for warps that go on by themselves: whichever of them gives up raises the status word (one warp's wait may run out
// and another's not, a moment later).
__device__ __forceinline__ bool mbar_wait_warp_or_report(uint64_t *bar, uint32_t parity, int32_t *status) {
  const bool ok = mbar_wait_warp(bar, parity);
  if (!ok && (threadIdx.x & 31) == 0) atomicMin(status, (int32_t)PACT_ERR_TIMEOUT);
  return ok;
}

// The same for a warp with more waits to come in a CTA that may have given up: once *abort is set nothing is asked for any more,
// and it does not wait a second for each of them.  (One lane looks: the answer has to be the warp's.  It looks when the first
// attempt has failed: 0.4 us of k_merge's 75 for 16 images of 2916 tokens, 0.5 with the look first.)
__device__ __forceinline__ bool mbar_wait_warp_unless(const int *abort, uint64_t *bar, uint32_t parity) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) ok = mbar_try_wait(bar, parity) || (!*const_cast<const volatile int *>(abort) && mbar_wait(bar, parity)) ? 1 : 0;
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}

}  // namespace pact
