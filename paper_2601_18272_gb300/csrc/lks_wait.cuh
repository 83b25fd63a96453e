// Bounded waits of the persistent kernels.
#pragma once

#include "lks_device.cuh"

namespace lks {

constexpr unsigned long long kSyncTimeoutNs = 1000000000ull;  // one second

__device__ __forceinline__ unsigned long long globaltimer_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// over(): called once per unsuccessful poll; true when the wait has lasted kSyncTimeoutNs or another
// CTA has given up (ST_SYNC_TIMEOUT in *status, which it sets). The clock and the status word are
// read every 64 polls only.
struct WaitLimit {
  unsigned long long t0 = 0;
  unsigned polls = 0;
  __device__ __forceinline__ bool over(int* status) {
    if (++polls & 63u) return false;
    if (*(volatile int*)status & ST_SYNC_TIMEOUT) return true;
    const unsigned long long now = globaltimer_ns();
    if (t0 == 0) t0 = now;
    if (now - t0 <= kSyncTimeoutNs) return false;
    atomicOr(status, ST_SYNC_TIMEOUT);
    return true;
  }
};

}  // namespace lks
