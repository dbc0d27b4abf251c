// Library-owned handle layouts (opaque to C callers).
#pragma once

#include <vector>

#include "seg_gather.cuh"

// The segmented graph of Algorithm 2, flattened: all subgraphs concatenated
// in segment order.  Subgraph row i (global row index over all segments)
// holds edges [row_ptr[i], row_ptr[i+1]) (stored flagged and padded in
// plan.colf) and its destination is idx_map[i].  blk[b*k + s] is the first
// (global) row of segment s whose destination is >= b*mB (block-major: a
// merge block's starts of all segments are contiguous); rows of segment s
// inside merge block b are [blk[b*k + s], blk[(b+1)*k + s]).
struct cg_segmented {
  int device = 0;
  int32_t V = 0;
  int64_t E = 0;
  int32_t k = 0;
  int32_t B = 0;
  int32_t nb = 0;
  int32_t mB = 0;              // destinations per warp of the merge (at most B, see merge_block)
  int32_t mnb = 0;             // merge blocks of mB destinations
  int64_t rows = 0;
  std::vector<int64_t> bounds, row_base, edge_base;  // host copies, k+1 each
  int32_t* idx_map = nullptr;  // [rows]; row_ptr and blk lie in the same allocation
  int32_t* row_ptr = nullptr;  // [rows+1] (builds and export; the gathers do not read it)
  int32_t* blk = nullptr;      // [(mnb+1)*k] block-major
  cg::SegPlan plan;            // flagged padded edges + chunk index + launch shape
  char* state = nullptr;         // one allocation that holds the arrays below
  void* interm = nullptr;        // [rows] 4-byte values (intermBuf)
  double* partials = nullptr;    // [2*nb] per-block FP64 partial sums
  unsigned* counter = nullptr;   // last-block detection
  double* dslot = nullptr;       // [4] FP64 iteration state (dangling ping-pong, scratch)
  float* rank_tmp = nullptr;     // [V] ping-pong for multi-iteration calls
  float* contrib_tmp = nullptr;  // [V]
  int64_t bytes = 0;
  // where a pass's count of changed labels goes, and its ticket (lp_run, from its
  // first call on)
  mutable unsigned long long* pin = nullptr;
  mutable unsigned long long ticket = 0;
};

// The plain pull baseline: the caller's CSR plus a merge-path tiling.
struct cg_plain {
  int device = 0;
  int32_t V = 0;
  int64_t E = 0;
  const int64_t* offsets = nullptr;  // caller-owned
  const int32_t* src = nullptr;      // caller-owned
  cg::TilePlan plan;
  float* acc = nullptr;          // [V] gathered sums
  double* partials = nullptr;    // [2*nb]
  unsigned* counter = nullptr;
  double* dslot = nullptr;       // [4]
  float* rank_tmp = nullptr;
  float* contrib_tmp = nullptr;
  int32_t nb = 0;
  int64_t bytes = 0;
};

namespace cg {
// Destinations per warp of the merge: the most, up to the caller's B and in
// steps of 32, with which the warps make whole waves of 40 per SM.  One warp's merge
// is a chain of dependent reads, so a small graph's time is that chain, and a last
// wave that is nearly empty costs as much as a full one.  48 warps (6 blocks) fit;
// counting on 40 was the best of 24, 32, 36, 40, 44 and 48 from 300 K to 33 M
// vertices (20 iterations with 48 and 40: 300 K 770 and 661 us, 1 M 1167 and 1073, 4
// M 2869 and 2762, 33 M 17.70 ms both), measured, not derived.  (The caller's B = 512
// itself put 20,011 vertices on 5 of 152 SMs: 11.0 us, 4.9 so.)  A block of hubs has
// rows in every one of the k segments: where that makes more than 3000 for one
// warp, up to three waves share them out.  One merge without that, and with 6000,
// 3000 and 1500: 1 M vertices, 40 segments 27.9, 16.8, 13.1, 13.0 us; 3 M, 9 segments
// 28.6, 28.4, 17.0, 14.2; 3 M, 40 segments 74.5, 32.7, 32.8, 32.9; 4 M, 7 segments
// 18.0, 18.4, 18.3, 15.1; 8 M the same with all.
int32_t merge_block(int32_t V, int32_t B, int32_t k, int sm_count);

// Validate an in-edge CSR on the device (offsets monotone from 0 to E, every
// source in [0, V)).  Synchronizes the stream.
int validate_csr(const int64_t* offsets, const int32_t* src, int32_t V, int64_t E,
                 cudaStream_t s);
}  // namespace cg
