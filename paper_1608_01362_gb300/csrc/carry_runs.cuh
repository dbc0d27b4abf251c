// Rows that span the pieces of work of a gather.
#pragma once

#include "gather.cuh"

namespace cg {

// Completion of the rows that span chunks: carry c belongs to row carry_row[c]
// (-1: none), and the carries of one row are consecutive (a run).  A warp
// takes 32 carries and finishes the runs that begin among them: those that
// also end there by one segmented scan, the last one by reading on, 128
// carries at a time, until its row ends.  The order is fixed: deterministic.
// (The run lists this replaces were made by the host from a copy of the rows,
// 0.7 ms of a new 65 M-edge graph.)
//
// Where a row has a thousand carries and more (a star's centre in a segment read
// through L1/L2), reading on is a long chain, 1.3 us per 128 of them.  Such a plan
// has the carries summed by tiles first (carry_tile_sums); tiles that lie within one
// row then stand for their carries.  A star of 1 M vertices, 7,813 carries in one row:
// 91 us for the fix-up, 10 with the tiles.
constexpr int kCarryTile = 256;
constexpr int kLongRun = 512;  // a plan has tile sums if one row has all of so many
                               // aligned carries

template <class Op>
__device__ __forceinline__ void carry_tile_sums(const int32_t* carry_row,
                                                const typename Op::T* carry, int64_t n,
                                                typename Op::T* __restrict__ tiles) {
  const int lane = threadIdx.x & 31;
  const int64_t step = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < n / kCarryTile;
       t += step) {
    const int64_t c = t * kCarryTile;
    const int32_t r = __ldca(carry_row + c);
    if (r < 0 || __ldca(carry_row + c + kCarryTile - 1) != r) continue;
    typename Op::T v = Op::identity();
#pragma unroll
    for (int u = 0; u < kCarryTile / 32; ++u) v = Op::op(v, __ldca(carry + c + 32 * u + lane));
#pragma unroll
    for (int o = 16; o; o >>= 1) v = Op::op(v, __shfl_xor_sync(0xffffffffu, v, o));
    if (lane == 0) tiles[t] = v;
  }
}

// TILES: tiles holds the carries' tile sums.
template <class Op, bool TILES = false>
__device__ __forceinline__ void fix_runs(const int32_t* carry_row,
                                         const typename Op::T* carry, int64_t n,
                                         typename Op::T* __restrict__ out,
                                         const typename Op::T* tiles = nullptr) {
  using T = typename Op::T;
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t step = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) << 5; c0 < n;
       c0 += step) {
    const int64_t c = c0 + lane;
    const int32_t r = c < n ? __ldca(carry_row + c) : -1;
    int32_t prev = __shfl_up_sync(kFull, r, 1), next = __shfl_down_sync(kFull, r, 1);
    if (lane == 0) prev = c0 > 0 ? __ldca(carry_row + c0 - 1) : -1;
    if (lane == 31) next = c0 + 32 < n ? __ldca(carry_row + c0 + 32) : -1;
    T S = r >= 0 ? carry[c] : Op::identity();
    int h = r < 0 || r != prev;  // a run begins (or none lies) here
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const T y = __shfl_up_sync(kFull, S, o);
      const int g = __shfl_up_sync(kFull, h, o);
      if (lane >= o) {
        if (!h) S = Op::op(y, S);
        h |= g;
      }
    }
    if (r >= 0 && h && next != r) out[r] = Op::op(S, out[r]);
    if (!__shfl_sync(kFull, (int)(r >= 0 && h && next == r), 31)) continue;
    const int32_t row = __shfl_sync(kFull, r, 31);
    T t = __shfl_sync(kFull, S, 31);
    bool more = true;
    for (int64_t b = c0 + 32; more;) {
      T v = Op::identity();
      if (TILES && b % kCarryTile == 0) {  // 128 tiles at a time, as far as they are the row's
        int64_t whole = 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int64_t q = b / kCarryTile + 32 * u + lane, i = q * kCarryTile;
          const unsigned m =
              __ballot_sync(kFull, i + kCarryTile <= n && __ldca(carry_row + i) == row &&
                                       __ldca(carry_row + i + kCarryTile - 1) == row);
          const int len = whole < 32 * u ? 0 : m == kFull ? 32 : __ffs(~m) - 1;
          if (lane < len) v = Op::op(v, __ldca(tiles + q));
          whole += len;
        }
        if (whole > 0) {
#pragma unroll
          for (int o = 16; o; o >>= 1) v = Op::op(v, __shfl_xor_sync(kFull, v, o));
          t = Op::op(t, v);
          b += whole * kCarryTile;
          continue;
        }
      }
      // (with tiles, up to the next multiple of 128, so that a tile's start is met)
      const int64_t end = TILES ? (b / 128 + 1) * 128 : b + 128;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        const int64_t i = b + 32 * u + lane;
        const unsigned m = __ballot_sync(kFull, i < n && __ldca(carry_row + (i < n ? i : 0)) == row);
        if (b + 32 * u >= end) continue;
        const int len = !more ? 0 : m == kFull ? 32 : __ffs(~m) - 1;
        if (lane < len) v = Op::op(v, carry[i]);
        more = more && len == 32;
      }
#pragma unroll
      for (int o = 16; o; o >>= 1) v = Op::op(v, __shfl_xor_sync(kFull, v, o));
      t = Op::op(t, v);
      b = end;
    }
    if (lane == 0) out[row] = Op::op(t, out[row]);
  }
}

}  // namespace cg
