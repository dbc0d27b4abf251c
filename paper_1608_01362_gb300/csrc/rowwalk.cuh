// Which row does an edge belong to?  A warp that takes consecutive edges of a
// CSR (or of any rows laid end to end) keeps the ends of 32 consecutive rows
// in its lanes and finds each edge's row among them with five shuffles; it
// moves on to the next 32 rows when its edges pass them, and searches the row
// offsets anew (32-ary, five or six dependent reads) only where those do not
// hold the edge, i.e. at its start and behind long runs of empty rows.
//
// Work is thus cut by edges, not rows: a hub row is spread over many warps, a
// thousand short rows share one, and the row lookup costs about 20
// instructions per 32 edges.  (The warp-per-row kernels this replaces left
// most lanes idle on short rows and held up one warp for a hub.)
#pragma once

#include "common.cuh"

namespace cg {

// Row ends of at most 2^31 - 1 edges; OffT is the stored offset type.
template <typename OffT>
struct RowWalk {
  const OffT* off;  // off[r]: first edge of row r, off[n] the total
  int32_t n;        // rows
  int32_t r0;       // first row of the window
  int32_t end;      // this lane's row end: off[r0 + lane + 1] (the total past row n)
  int32_t start;    // off[r0]
  int32_t ahead;    // the same of the next 32 rows, read ahead

  __device__ __forceinline__ int32_t end_of(int32_t r) const {  // row r's end, for this lane's r
    return (int32_t)__ldg(off + min((int64_t)r + 1, (int64_t)n));
  }
  __device__ __forceinline__ void window(int32_t r) {
    const int lane = threadIdx.x & 31;
    r0 = r;
    start = (int32_t)__ldg(off + r);
    end = end_of((int32_t)min((int64_t)r + lane, (int64_t)n));
    ahead = end_of((int32_t)min((int64_t)r + 32 + lane, (int64_t)n));
  }
  __device__ __forceinline__ void advance() {
    const int lane = threadIdx.x & 31;
    start = __shfl_sync(0xffffffffu, end, 31);
    end = ahead;
    r0 = (int32_t)min((int64_t)r0 + 32, (int64_t)n);
    ahead = end_of((int32_t)min((int64_t)r0 + 32 + lane, (int64_t)n));
  }

  // window at the row of edge e (uniform in the warp): the last r with off[r] <= e
  __device__ __forceinline__ void seek(int32_t e) {
    const int lane = threadIdx.x & 31;
    int32_t lo = 0, hi = n;  // off[lo] <= e < off[hi]
    while (hi - lo > 1) {
      const int32_t step = (hi - lo + 32) / 33;  // probes lo + step, lo + 2 step, ...
      const int64_t p = (int64_t)lo + (int64_t)step * (lane + 1);
      const bool le = p < hi && (int32_t)__ldg(off + p) <= e;
      const int c = __popc(__ballot_sync(0xffffffffu, le));
      const int64_t nh = (int64_t)lo + (int64_t)step * (c + 1);
      lo += step * c;
      if (nh < hi) hi = (int32_t)nh;
    }
    window(lo);
  }

  // Row of this lane's edge e and the row's first edge; lanes' edges ascend
  // with the lane, ok tells which lanes have one (a prefix of the warp).
  __device__ __forceinline__ int32_t row_of(int32_t e, bool ok, int32_t* row_start) {
    const unsigned full = 0xffffffffu;
    int32_t row = 0, st = 0;
    unsigned todo = __ballot_sync(full, ok);
    while (todo) {
      const int first = __ffs(todo) - 1;
      const int32_t ef = __shfl_sync(full, e, first);
      if (ef >= __shfl_sync(full, end, 31)) {  // past the window
        advance();
        if (ef >= __shfl_sync(full, end, 31)) seek(ef);
      }
      int j = 0;  // rows of the window that end at or before e
#pragma unroll
      for (int s = 16; s; s >>= 1)
        if (__shfl_sync(full, end, j + s - 1) <= e) j += s;
      // j = 31 may also mean that all 32 end before e
      const int32_t ej = __shfl_sync(full, end, j);
      const int32_t sj = __shfl_sync(full, end, j > 0 ? j - 1 : 0);
      const bool mine = ((todo >> (threadIdx.x & 31)) & 1u) && e < ej;
      if (mine) {
        row = r0 + j;
        st = j > 0 ? sj : start;
      }
      todo &= ~__ballot_sync(full, mine);
    }
    *row_start = st;
    return row;
  }
};

}  // namespace cg
