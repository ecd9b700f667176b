// bounded_wait.cuh -- waiting for asynchronous copies without the risk of
// waiting for ever.
#pragma once

namespace sphynx {

constexpr int kWaitTries = 1 << 22;                 // polls, each a bounded hardware wait of its own
constexpr long long kWaitCycles = 2000000000ll;     // and about a second of SM clock

// true once phase 0 of the mbarrier at shared address bar32 has completed, false
// when kWaitTries polls or kWaitCycles were not enough
__device__ __forceinline__ bool bounded_wait(unsigned bar32) {
  const long long t0 = clock64();
  for (int tries = 0; tries < kWaitTries; ++tries) {
    unsigned ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], 0;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok)
                 : "r"(bar32)
                 : "memory");
    if (ok) return true;
    if (clock64() - t0 > kWaitCycles) return false;
  }
  return false;
}

// For whole warps: bounded_wait, and where it gives up *fault (host memory) is
// set, which the handle's next call turns into an error.  The copies may still
// be in flight then and must not find this block's shared memory in other hands,
// so that a second wait, as long as the first, comes before the return; the
// caller ends without touching the data either way.
__device__ __forceinline__ bool bounded_wait_or_fault(unsigned bar32, int *fault) {
  if (__all_sync(0xffffffffu, bounded_wait(bar32))) return true;
  *static_cast<volatile int *>(fault) = 1;
  __threadfence_system();
  (void)bounded_wait(bar32);
  return false;
}

}  // namespace sphynx
