// Collaborative filtering through segments of the neighbour side (cf_seg.cu).
#pragma once

#include "ranges.cuh"

namespace cg {

// One side's pieces: runs of at most kCfSegPiece consecutive ratings of one
// vertex whose neighbours lie in one segment, grouped into warp tasks.
struct CfSegments {
  int32_t k = 0;               // segments of `width` neighbour rows (0: not used)
  int32_t width = 0;
  int32_t ntasks = 0;
  int64_t npieces = 0;
  int64_t nslots = 0;          // ntasks x pieces per task
  char* slab = nullptr;        // one allocation that holds the arrays below
  int4* recs = nullptr;        // [nslots] (first rating, ratings, vertex, -); unused: 0 ratings
  int32_t* slots = nullptr;    // [npieces] a vertex's pieces' slots, in rating order
  int64_t* poff = nullptr;     // [n+1] first piece of each vertex
  int32_t* seg_task = nullptr; // [k+1] first task of each segment
  int32_t* blk_task = nullptr; // [grid+1]
  unsigned* next = nullptr;    // [grid]
  int grid = 0;
  int64_t bytes = 0;
};

// Lay out one side (n vertices, their CSR over nn neighbours, K dimensions).
// Leaves k = 0 where the earlier gather is the better one (see cf_seg.cu).
// Synchronizes.
int cf_seg_build(CfSegments* c, int64_t n, int64_t nn, int64_t R, int K, const int64_t* off,
                 const int32_t* nbr, cudaStream_t s);
void cf_seg_free(CfSegments* c);

// Piece gradients of one side into gpart[slot][K]; sse (side 0): the squared
// errors' sum.  self / other: the two sides' factors in their storage.
int cf_seg_gather(const CfSegments& c, int K, int precision, int64_t nn, const int32_t* nbr,
                  const uint8_t* rate, const void* self, const void* other, float* gpart,
                  bool with_sse, double* partials, unsigned* counter, double* sse,
                  cudaStream_t s);

}  // namespace cg
