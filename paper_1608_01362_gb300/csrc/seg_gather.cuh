// Segment processing (Algorithm 3) over the flattened segmented graph.
//
// Edge layout ("colf"): the subgraphs' source IDs, segment after segment,
// each segment starting on an 8-entry (32-byte) boundary; bit 31 of an entry
// marks the last edge of its subgraph row.  Every subgraph row has at least
// one edge, so row i is the (i+1)-th flagged edge: the gather needs no row
// pointers at all.
//
// Work unit of the segments read through L1/L2: a warp owns a chunk of 128 or 256
// consecutive edges of one segment (4 or 8 per lane, by the number of such edges);
// lane l holds edges [IPL l, IPL (l + 1)) of it (16-byte streaming loads).  Lanes fold
// their values sequentially, emit every row that starts and ends inside them, and a
// warp-wide segmented scan over the lanes' open-row parts completes each lane's first
// row.  The row still open at the chunk's end goes to carry[chunk], folded in
// afterwards in chunk order.  No shared staging of edges and no block barriers
// between chunks.  The staged segments' unit is the warp task of a layout of their
// own (staged_stream.cuh).
//
// Launches of a pass, each where there is something for it:
//   staged    the leading segments that fit an SM's shared memory (after clustering,
//             the hot head: the paper's cache-sized segment, sized here to on-chip
//             shared memory): each block copies its current segment's source values
//             into shared memory and every read of the segment is served from there.
//             A block owns a contiguous range of tasks, which meets one or two
//             segments, and helps with the fullest range when its own runs dry
//             (ranges.cuh).
//   affine    with the segment-affine plan: the table-sized segments behind the head,
//             one block per segment, handed out by a counter.
//   cached    the remaining segments, through L1/L2, without shared memory, which
//             leaves the whole on-chip store to the L1 cache.  Blocks take block-sized
//             groups of chunks round robin, in segment order.
//   fix-up    rows that span chunks or full pieces (carry_runs.cuh).
// With the overlap one launch serves the staged and the cached segments.
#pragma once

#include <vector>

#include "gather.cuh"

namespace cg {

constexpr uint32_t kRowEndFlag = 0x80000000u;
constexpr int kMaxChunkEdges = 512;  // padding behind the edges: a chunk may read past the end

struct SegPlan {
  int k = 0;
  int64_t E = 0, rows = 0, nchunks = 0;
  uint32_t* colf = nullptr;        // [colf_len] flagged, padded segment-local sources
  uint8_t* cs = nullptr;           // staged segments' edge stream (staged_stream.cuh)
  int64_t cs_cap = 0;
  uint4* desc = nullptr;           // one descriptor per staged task
  void* lent = nullptr;     // scratch that a caller of seg_plan_finish has at hand
  size_t lent_bytes = 0;
  int32_t* seg_task = nullptr;     // [k+1] first staged task of each segment
  std::vector<int32_t> h_seg_task;
  int32_t head_tasks = 0;          // tasks of the segments [0, m)
  int32_t* blk_task = nullptr;     // [grid+1] first task of each staged block's range
  int64_t colf_len = 0;
  int64_t* meta = nullptr;         // one allocation: row_base, edge_base, cstart, bounds (k+1
                                   // each), then the segments' arrays below
  int64_t* seg_cstart = nullptr;   // [k]   first colf entry of each segment
  int32_t* seg_E = nullptr;        // [k]   edges of each segment
  int64_t* seg_chunk = nullptr;    // [k+1] first global chunk of each segment
  int32_t* seg_ctile = nullptr;    // [k+1] first L1/L2 block-group of each segment
  int32_t* seg_lo = nullptr;       // [k]   first source of each segment
  int32_t* seg_tab = nullptr;      // [k]   table entries used for each segment
  // carries: one per L1/L2 chunk, then one per full piece of a long staged row; one allocation
  int32_t* first_row = nullptr;    // subgraph row of each L1/L2 chunk's first edge
  int32_t* carry_row = nullptr;    // [ncarry] the row a carry belongs to (-1: none)
  void* carry = nullptr;           // [ncarry] 4-byte values
  void* carry_tiles = nullptr;     // [ncarry / 256] sums of them, for plans with long_runs
  int64_t ncarry = 0, carry_cap = 0;
  bool long_runs = false;          // a row has hundreds of carries (carry_runs.cuh)
  const int32_t* rp32 = nullptr;   // subgraph row starts (owned by the handle)
  std::vector<int64_t> h_cstart, src_bounds, edge_base, row_base;
  bool ready = false;       // configured (false where a configuration failed half way)
  int threads = 1024;       // staged-segment launch shape
  int ctas_per_sm = 1;
  int tab_cap = 0;          // table entries of the staged launch (its largest segment)
  int table_request = 0;    // the capacity asked for
  int m = 0;                // segments [0, m) are staged in shared memory (all blocks sweep them)
  int m2 = 0;               // segments [m, m2): staged too, one block per segment (affine)
  double affine_head = 0.0;  // > 0: head threshold (edges per source) of the segment-affine
                            // plan; the table-sized segments after the head go one per block
  int cached_ipl = 8;          // edges per lane of an L1/L2 chunk
  int64_t ncached = 0;         // L1/L2 chunks
  int grid_affine = 0;      // blocks of the segment-affine launch
  int64_t n_ctiles = 0;     // block-groups of the L1/L2 launch
  int grid = 0;             // staged launch blocks
  unsigned* counter = nullptr;  // next L1/L2 chunk (overlap), next segment-affine segment, blocks
                                // finished of either, tasks taken of each staged block's range;
                                // zero between launches (the last block of each clears them)
  unsigned* found = nullptr;    // a word for the configuration
  int overlap_request = 0;  // warps per block given to the L1/L2 segments (0: two launches)
  int overlap = 0;          // the same, in effect (0 when one kind of segment is absent)
  int grid_l2 = 0;          // unstaged launch blocks (1024 threads, 2 per SM)
};

// Largest shared table (entries, multiple of 32) for `ctas` blocks per SM.
int seg_table_capacity(int ctas);

// Allocate a plan for E edges in k segments (colf and the segments' arrays;
// the caller fills colf and meta's row_base), then, with the rows known (rp32:
// their first edges, kept by the handle), choose the default launch shape.
// Both synchronize.
int seg_plan_alloc(int64_t E, int k, const std::vector<int64_t>& edge_base,
                   const std::vector<int64_t>& src_bounds, SegPlan* p, cudaStream_t s);
int seg_plan_finish(SegPlan* p, const int32_t* rp32, int64_t rows,
                    const std::vector<int64_t>& row_base, cudaStream_t s);

// Launch shape: threads per block (512 or 1024), blocks per SM, table size
// (-1: the capacity; 0: none).  Synchronizes the stream.  CG_ERR_INVALID_ARG changes
// nothing; after another error no gather runs until a configuration succeeds.
int seg_plan_configure(SegPlan* p, int threads, int ctas_per_sm, int tab_vertices,
                       cudaStream_t s);

// Lay out the staged segments [0, m2): their tasks, descriptors and stream (pad:
// the table entry that holds the identity).  The carries of the full pieces of
// rows longer than kStagedMost follow the first carry_base ones; their rows are
// written to carry_row.  Synchronizes.
// place (optional): where each row's sum goes, below 65535, in the place of its
// position in its window (the tasks' base row is then 0).
int staged_build(SegPlan* p, int m2, int pad, int64_t carry_base, cudaStream_t s,
                 const int32_t* place = nullptr);
// Room for n carries (their contents are lost when it grows).
int seg_plan_carries(SegPlan* p, int64_t n);

void seg_plan_free(SegPlan* p);
int64_t seg_plan_bytes(const SegPlan& p);

// Recover the unpadded source array (flags cleared) for export.
int seg_plan_export_col(const SegPlan& p, const int32_t* rp, int32_t* col, cudaStream_t s);

// Launch phases of one pass (all by default): the staged launch, the L1/L2
// launch (with the segment-affine staged launch before it, when configured)
// and the carry fix-up, in that order.  With the overlap in effect one
// launch serves both kinds of segment: it runs for kPhaseStaged and
// kPhaseCached launches nothing.
constexpr int kPhaseStaged = 1, kPhaseCached = 2, kPhaseFixup = 4, kPhaseAll = 7;

template <class Op>
int run_seg_gather(const SegPlan& p, const typename Op::T* x, int32_t nx, typename Op::T* out,
                   cudaStream_t s, int phases = kPhaseAll);

}  // namespace cg
