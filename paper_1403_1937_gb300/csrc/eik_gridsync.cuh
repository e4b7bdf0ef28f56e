// Grid-wide exchange of reduction partials inside one cooperative kernel
// (internal).  Every block publishes one or more tagged values per exchange
// and reads those of all blocks itself, so a reduction costs one store and
// one load round trip through L2 (no counter, no second pass over partials):
// a value is split into two 64-bit words, each carrying the exchange's 32-bit
// tag beside half of the value, and a reader polls both words until both tags
// match.  Slots alternate between two sets by the tag's parity: a block can
// be at most one exchange ahead of another, so the set it writes has been
// read by everybody.  Polls are bounded on %globaltimer; a block that waits
// in vain reports a fault and the kernel returns.
#pragma once

#include <stdint.h>

namespace eik {

constexpr unsigned long long kSyncWaitNs = 1000ull * 1000 * 1000;   // 1 s

// Values per exchange and block that a buffer has room for.
constexpr int kSyncVals = 2;

__device__ __forceinline__ unsigned long long sync_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Most blocks that take part (a warp reads five slots per lane), and the size
// of a solver's message buffer.
constexpr int kSyncBlocks = 160;
constexpr size_t kSyncBytes = sizeof(unsigned long long) * 2 * kSyncVals * 2 * kSyncBlocks;

// A double in two words, each with the 32-bit tag.
__device__ __forceinline__ void tagged_put(unsigned long long *slot, unsigned tag, double x) {
  const unsigned long long u = (unsigned long long)__double_as_longlong(x);
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(slot),
               "l"(t | (u & 0xffffffffull)), "l"(t | (u >> 32))
               : "memory");
}
__device__ __forceinline__ bool tagged_try(const unsigned long long *slot, unsigned tag,
                                           double *x) {
  unsigned long long lo, hi;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
               : "=l"(lo), "=l"(hi)
               : "l"(slot)
               : "memory");
  *x = __longlong_as_double((long long)((hi << 32) | (lo & 0xffffffffull)));
  return (unsigned)(lo >> 32) == tag && (unsigned)(hi >> 32) == tag;
}
// Bounded wait for one tagged value.
__device__ __forceinline__ bool tagged_wait(const unsigned long long *slot, unsigned tag,
                                            double *x) {
  if (tagged_try(slot, tag, x)) return true;
  unsigned long long t0 = 0;
  for (unsigned spins = 1;; ++spins) {
    if (tagged_try(slot, tag, x)) return true;
    if ((spins & 255u) == 0u) {
      const unsigned long long t = sync_now();
      if (t0 == 0) t0 = t;
      else if (t - t0 > kSyncWaitNs) return false;
    }
  }
}

__device__ __forceinline__ unsigned long long *sync_slot(unsigned long long *msg, unsigned tag,
                                                         int v, int b, int nblk) {
  return msg + 2 * ((size_t)((tag & 1u) * kSyncVals + v) * nblk + b);
}

__device__ __forceinline__ void sync_put(unsigned long long *msg, unsigned tag, int v, int b,
                                         int nblk, double x) {
  tagged_put(sync_slot(msg, tag, v, b, nblk), tag, x);
}

// Waits for value v of the blocks b0, b0 + 32, ... (at most N of them, those
// below nblk); x[j] = 0 past the end.  False when the wait ran out.
template <int N>
__device__ __forceinline__ bool sync_wait(unsigned long long *msg, unsigned tag, int v, int b0,
                                          int nblk, double (&x)[N]) {
  unsigned long long t0 = 0;
  for (unsigned spins = 1;; ++spins) {
    bool ok = true;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      x[j] = 0.0;
      if (b0 + 32 * j < nblk)
        ok = tagged_try(sync_slot(msg, tag, v, b0 + 32 * j, nblk), tag, &x[j]) && ok;
    }
    if (ok) return true;
    if ((spins & 255u) == 0u) {
      const unsigned long long t = sync_now();
      if (t0 == 0) t0 = t;
      else if (t - t0 > kSyncWaitNs) return false;
    }
  }
}

}  // namespace eik
