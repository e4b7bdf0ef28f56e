// Grid-wide sums inside one cooperative kernel, and values passed from block
// to block (internal).
//
// A sum: every block stores its partials in slots of its own, adds one to a
// counter (release), waits until the counter has every block's arrival
// (acquire, one thread), and reads all partials itself, so that all blocks add
// the same numbers in the same order.  Measured on 152 blocks: 2,700 cycles
// from arrival to the last partial read.  (Partials that carry a tag and are
// polled by every block need no counter, but 152 readers polling lines that
// eight blocks write took 5,500 to 8,000 cycles; a leader block that adds and
// publishes took 2,600, and needs a block or warp with nothing else to do.)
// Slots alternate between two sets by the exchange's parity: a block can be at
// most one exchange ahead of another, so the set it writes has been read by
// everybody.
//
// A value for one other block is stored as two 64-bit words, each with a
// 32-bit tag beside half of the value, which the reader polls until both tags
// match: no fence, no barrier.
//
// Every wait is bounded on %globaltimer; a block that waits in vain reports a
// fault and the kernel returns.
#pragma once

#include <math.h>
#include <stdint.h>

namespace eik {

constexpr unsigned long long kSyncWaitNs = 1000ull * 1000 * 1000;   // 1 s

// Partials per exchange and block, and most blocks that take part (a warp
// reads five slots per lane).
constexpr int kSyncVals = 3;
constexpr int kSyncBlocks = 160;
// A solver's buffer: a 128-byte line with the counter (its first 32 bits,
// zeroed before every launch) and, from the second word on, what a solver keeps
// between launches; then the slots.
constexpr int kSyncSlot0 = 16;
constexpr size_t kSyncBytes =
    sizeof(unsigned long long) * (kSyncSlot0 + 2 * kSyncVals * kSyncBlocks);

__device__ __forceinline__ unsigned long long sync_now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

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

__device__ __forceinline__ double *sync_slot(unsigned long long *msg, unsigned tag, int v, int b) {
  return reinterpret_cast<double *>(msg) + kSyncSlot0 + ((tag & 1u) * kSyncVals + v) * kSyncBlocks +
         b;
}
// Block b's partial v of exchange `tag`; sync_arrive by the same thread follows.
__device__ __forceinline__ void sync_put(unsigned long long *msg, unsigned tag, int v, int b,
                                         double x) {
  asm volatile("st.relaxed.gpu.global.f64 [%0], %1;" ::"l"(sync_slot(msg, tag, v, b)), "d"(x)
               : "memory");
}
__device__ __forceinline__ void sync_arrive(unsigned long long *msg) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(msg) : "memory");
}
// Warp 0: waits until the counter has `target` arrivals (those of all blocks
// in all exchanges of this launch so far).  False when the wait ran out.
__device__ __forceinline__ bool sync_wait(unsigned long long *msg, unsigned target) {
  int ok = 1;
  if ((threadIdx.x & 31) == 0) {
    unsigned long long t0 = 0;
    for (unsigned spins = 1;; ++spins) {
      unsigned c;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(c) : "l"(msg) : "memory");
      if (c >= target) break;
      if ((spins & 255u) == 0u) {
        const unsigned long long t = sync_now();
        if (t0 == 0) t0 = t;
        else if (t - t0 > kSyncWaitNs) {
          ok = 0;
          break;
        }
      }
    }
  }
  // (the shuffle orders no memory accesses: the other lanes' reads of the
  // partials come after lane 0's acquire by this barrier)
  __syncwarp();
  return __shfl_sync(0xffffffffu, ok, 0) != 0;
}
// Warp 0, after sync_wait: partial v of the blocks lane, lane + 32, ... (0 past
// the last).
__device__ __forceinline__ void sync_get(unsigned long long *msg, unsigned tag, int v, int nblk,
                                         double (&x)[kSyncBlocks / 32]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int j = 0; j < kSyncBlocks / 32; ++j) {
    x[j] = 0.0;
    if (lane + 32 * j < nblk)
      asm volatile("ld.relaxed.gpu.global.f64 %0, [%1];"
                   : "=d"(x[j])
                   : "l"(sync_slot(msg, tag, v, lane + 32 * j))
                   : "memory");
  }
}
// Their sum over the warp, in a fixed order, in all lanes.
__device__ __forceinline__ double sync_sum(const double (&x)[kSyncBlocks / 32]) {
  double s = ((x[0] + x[1]) + (x[2] + x[3])) + x[4];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  return s;
}

// a / b for finite a >= 0 and b > 0 to within three units in the last place (a
// step length needs no more): a single-precision reciprocal y of b's mantissa m
// and the first terms of 1 / m = y / (1 - e) = y (1 + e + e^2 + ...), e = 1 - m y
// (M. J. Flynn, On division by functional iteration, IEEE Trans. Computers C-19,
// 1970).  A dependent FP64 operation takes about 90 cycles here; this has five.
__device__ __forceinline__ double quotient(double a, double b) {
  const int hb = __double2hiint(b);
  const int eb = (hb >> 20) - 1023;
  // subnormal (its quotient with a mantissa would be rounded there) or near the top
  if (eb <= -1023 || eb >= 1023 || (__double2hiint(a) >> 20) == 0) return a / b;
  const double m = __hiloint2double((hb & 0x000fffff) | 0x3ff00000, __double2loint(b));
  const double y = (double)(1.0f / (float)m);
  const double e = fma(-m, y, 1.0);
  const double q = a * fma(y, fma(e, e, e), y);
  // q 2^-eb: on the exponent bits unless that leaves the normal range
  const int hq = __double2hiint(q), eq = (hq >> 20) - eb;
  if (eq <= 0 || eq >= 2047 || (hq >> 20) == 0) return scalbn(q, -eb);
  return __hiloint2double(hq - (eb << 20), __double2loint(q));
}

// Barrier among the first n threads of a block.
__device__ __forceinline__ void bar_first(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}

}  // namespace eik
