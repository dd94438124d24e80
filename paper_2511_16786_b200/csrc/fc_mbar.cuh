// Shared-memory barriers (mbarrier) with bounded waits: the decoding kernel's ring, and the self test of the waits.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace mbar {

constexpr unsigned kSuspendNs = 2000u;       // a blocking test of an mbarrier sleeps at most about this long
constexpr unsigned kSpinLimit = 1u << 17;    // such tests before a wait gives up (a quarter of a second)

__device__ __forceinline__ unsigned address(const void *p) { return (unsigned)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void init(unsigned long long *bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(address(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void init_done() { asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory"); }
__device__ __forceinline__ void expect_tx(unsigned long long *bar, unsigned bytes) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n}\n"
               ::"r"(address(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void arrive(unsigned long long *bar) {
  asm volatile("{\n .reg .b64 st;\n mbarrier.arrive.shared::cta.b64 st, [%0];\n}\n" ::"r"(address(bar)) : "memory");
}
// One potentially blocking test: the thread sleeps until the phase completes or a hardware time limit passes.
__device__ __forceinline__ bool test(unsigned long long *bar, unsigned parity) {
  unsigned ok;
  asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n selp.u32 %0, 1, 0, p;\n}\n"
               : "=r"(ok) : "r"(address(bar)), "r"(parity), "r"(kSuspendNs) : "memory");
  return ok != 0u;
}
// Bounded wait of one thread; false = gave up.
__device__ __forceinline__ bool wait(unsigned long long *bar, unsigned parity, unsigned limit = kSpinLimit) {
  for (unsigned it = 0; it < limit; ++it)
    if (test(bar, parity)) return true;
  return false;
}
// Bounded wait of a whole warp: every lane waits (and so sees what the barrier guards), and all get one verdict, false if
// any lane gave up.  The warp's collective instructions may follow; a lane must not act on a verdict of its own.
__device__ __forceinline__ bool wait_warp(unsigned long long *bar, unsigned parity, unsigned limit = kSpinLimit) {
  return __all_sync(0xffffffffu, wait(bar, parity, limit)) != 0;
}

// A ring of S stages, item i in stage i % S: waits (bounded, S limits at most) for the loads of the last items of `issued`,
// each of which is the last one its stage was given.  Whoever issued loads into a block's shared memory calls this before
// it ends, whatever the consumers did: a block that has gone may have its memory given to another one.
template <int S>
__device__ __forceinline__ bool drain(unsigned long long (&full)[S], int issued, unsigned limit = kSpinLimit) {
  bool landed = true;
  for (int i = issued > S ? issued - S : 0; i < issued; ++i) landed &= wait(&full[i % S], (unsigned)(i / S) & 1u, limit);
  return landed;
}

}  // namespace mbar
