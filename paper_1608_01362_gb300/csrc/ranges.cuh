// Work shared by contiguous ranges: block b owns tasks [first[b], first[b+1])
// (equal stretches of the work), takes half of what is left of its range at a
// time, and when that runs dry half of what is left of the fullest range.
// Tasks sorted by the shared-memory table they need then meet one or two
// tables per block, and the blocks still finish together.  No block waits for
// another.
#pragma once

#include "common.cuh"

namespace cg {

struct RangeShare {
  const int32_t* first;  // [grid+1]
  unsigned* next;        // [grid] tasks taken of each range (zero before the launch)
};
struct RangeSlots {  // a block's shared words
  int32_t lo, hi;
  unsigned fullest;
};

constexpr int kStealMin = 64;  // a range with fewer tasks left is not worth a table copy

#ifdef __CUDACC__

// Barrier among threads [0, nt) of the block: the whole block, or named
// barrier 1 when only some of its warps take part.
__device__ __forceinline__ void group_sync(int nt) {
  if (nt == (int)blockDim.x)
    __syncthreads();
  else
    asm volatile("bar.sync 1, %0;" ::"r"(nt) : "memory");
}

// The next tasks [*t, *hi) for threads [0, nt) of the block (v: the range being
// worked on, blockIdx.x at first); false when every range is used up.
__device__ __forceinline__ bool next_range(const RangeShare& sh, int nt, RangeSlots* slots, int* v,
                                           int32_t* t, int32_t* hi) {
  const int tid = threadIdx.x;
  for (;;) {
    group_sync(nt);  // everyone is done with the previous piece and the slots
    if (tid == 0) {
      const int32_t b0 = sh.first[*v], n = sh.first[*v + 1] - b0;
      const int32_t taken = (int32_t)*(volatile unsigned*)(sh.next + *v);
      const int32_t sz = max((n - taken) / 2, kStealMin);
      const int32_t lo = taken < n ? (int32_t)atomicAdd(sh.next + *v, (unsigned)sz) : n;
      slots->lo = b0 + min(lo, n);
      slots->hi = b0 + min(lo + sz, n);
      slots->fullest = 0u;
    }
    group_sync(nt);
    *t = slots->lo;
    *hi = slots->hi;
    if (*t < *hi) return true;
    for (int b = tid; b < (int)gridDim.x; b += nt) {
      const int32_t left =
          sh.first[b + 1] - sh.first[b] - (int32_t)*(volatile unsigned*)(sh.next + b);
      if (left >= kStealMin)
        atomicMax(&slots->fullest, ((unsigned)min(left, 0x1FFFFF) << 11) | (unsigned)b);
    }
    group_sync(nt);
    if (slots->fullest == 0u) return false;
    *v = (int)(slots->fullest & 0x7FFu);
  }
}

// Which of m segments holds task t (first[q]: segment q's first task, ascending).
__device__ __forceinline__ int segment_of_task(const int32_t* first, int m,
                                               int32_t t) {
  const int lane = threadIdx.x & 31;
  int s = 0;  // segments whose tasks all precede t
  for (int i = 0; i < m; i += 32) {
    const unsigned bal =
        __ballot_sync(0xffffffffu, i + lane < m && __ldca(first + i + lane + 1) <= t);
    s += __popc(bal);
    if (bal != 0xffffffffu) break;
  }
  return s;
}

#endif  // __CUDACC__

}  // namespace cg
