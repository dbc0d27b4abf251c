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

// OffT is the stored offset type, PosT holds an edge's place: 32 bits below 2^31
// edges (rows that begin behind the last edge walked are taken to begin there).
// CHAINED: for kernels that are launched chained.
template <typename OffT, typename PosT = int32_t, bool CHAINED = false>
struct RowWalk {
  static __device__ __forceinline__ OffT load(const OffT* p) {
    return CHAINED ? __ldca(p) : __ldg(p);
  }
  const OffT* off;  // off[r] - origin: first edge of row r < n
  int32_t n;        // rows
  PosT total;       // edges walked, the end of row n - 1
  PosT origin;
  int32_t r0;       // first row of the window
  PosT start;       // its first edge
  PosT end;         // this lane's row end: that of row r0 + lane (the total past row n - 1)
  PosT ahead;       // the same of the next 32 rows, read ahead

  __device__ __forceinline__ RowWalk(const OffT* o, int32_t rows, PosT edges, PosT org = 0)
      : off(o), n(rows), total(edges), origin(org), r0(0), start(0), end(0), ahead(0) {}

  __device__ __forceinline__ PosT first_of(int64_t r) const {
    if (r >= n) return total;
    const OffT at = load(off + r) - (OffT)origin;
    return at < (OffT)total ? (PosT)at : total;
  }
  __device__ __forceinline__ void window(int32_t r) {
    const int lane = threadIdx.x & 31;
    r0 = r;
    start = first_of(r);
    end = first_of((int64_t)r + lane + 1);
    ahead = first_of((int64_t)r + lane + 33);
  }
  __device__ __forceinline__ void advance() {
    const int lane = threadIdx.x & 31;
    start = __shfl_sync(0xffffffffu, end, 31);
    end = ahead;
    r0 = (int32_t)min((int64_t)r0 + 32, (int64_t)n);
    ahead = first_of((int64_t)r0 + lane + 33);
  }

  // window at the row of edge e (uniform in the warp): the last r with off[r] <= e
  __device__ __forceinline__ void seek(PosT e) {
    const int lane = threadIdx.x & 31;
    int32_t lo = 0, hi = n;  // row lo begins at or before e, row hi behind it
    while (hi - lo > 1) {
      // probes lo + step, lo + 2 step, ... (unsigned: hi - lo goes up to 2^31 - 1)
      const int32_t step = (int32_t)(((uint32_t)(hi - lo) + 32u) / 33u);
      const int64_t p = (int64_t)lo + (int64_t)step * (lane + 1);
      const bool le = p < hi && load(off + p) - (OffT)origin <= (OffT)e;
      const int c = __popc(__ballot_sync(0xffffffffu, le));
      const int64_t nh = (int64_t)lo + (int64_t)step * (c + 1);
      lo += step * c;
      if (nh < hi) hi = (int32_t)nh;
    }
    window(lo);
  }

  // Row of this lane's edge e, the row's first edge and its end; lanes' edges
  // ascend with the lane, ok tells which lanes have one (a prefix of the warp).
  __device__ __forceinline__ int32_t row_of(PosT e, bool ok, PosT* row_start, PosT* row_end) {
    const unsigned full = 0xffffffffu;
    int32_t row = 0;
    PosT st = 0, en = 0;
    unsigned todo = __ballot_sync(full, ok);
    while (todo) {
      const int first = __ffs(todo) - 1;
      const PosT ef = __shfl_sync(full, e, first);
      if (ef >= __shfl_sync(full, end, 31)) {  // past the window
        advance();
        if (ef >= __shfl_sync(full, end, 31)) seek(ef);
      }
      int j = 0;  // rows of the window that end at or before e
#pragma unroll
      for (int s = 16; s; s >>= 1)
        if (__shfl_sync(full, end, j + s - 1) <= e) j += s;
      // j = 31 may also mean that all 32 end before e
      const PosT ej = __shfl_sync(full, end, j);
      const PosT sj = __shfl_sync(full, end, j > 0 ? j - 1 : 0);
      const bool mine = ((todo >> (threadIdx.x & 31)) & 1u) && e < ej;
      if (mine) {
        row = r0 + j;
        st = j > 0 ? sj : start;
        en = ej;
      }
      todo &= ~__ballot_sync(full, mine);
    }
    *row_start = st;
    *row_end = en;
    return row;
  }
};

// The same where every row has an edge (a list of such rows): 32 consecutive
// edges' row ends are then one bit mask, put together with one reduction from
// the window's ends, and a lane's row is a population count away: about 15
// instructions per 32 edges, no search.
struct DenseWalk {
  RowWalk<int32_t, int32_t, true> w;
  int32_t row;    // row of the next batch's first edge

  __device__ __forceinline__ DenseWalk(const int32_t* pos, int32_t rows, int32_t edges,
                                       int32_t origin = 0)
      : w(pos, rows, edges, origin), row(0) {}

  __device__ __forceinline__ void seek(int32_t e) {
    w.seek(e);
    row = w.r0;
  }
  // Row ends among the 32 edges from e on (bit q: edge e + q ends its row), and
  // this lane's row; the walk moves on behind them.
  __device__ __forceinline__ uint32_t batch(int32_t e, int32_t* lane_row) {
    const int lane = threadIdx.x & 31;
    const uint32_t a = (uint32_t)(w.end - 1 - e), b = (uint32_t)(w.ahead - 1 - e);
    // past the last row every end is the total: one bit for all of them
    const uint32_t bits = (a < 32u ? 1u << a : 0u) | (b < 32u ? 1u << b : 0u);
    const uint32_t ends = __reduce_or_sync(0xffffffffu, bits);
    *lane_row = row + __popc(ends & ((1u << lane) - 1u));
    row += __popc(ends);
    if (row - w.r0 >= 32) w.advance();
    return ends;
  }
};

}  // namespace cg
