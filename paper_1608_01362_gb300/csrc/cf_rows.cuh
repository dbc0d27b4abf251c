// Collaborative filtering: pieces of one side's ratings and their gather
// (cf_rows.cu).
#pragma once

#include "common.cuh"

namespace cg {

// One side's pieces: consecutive ratings of one vertex, at most `most` of them,
// in warp tasks of about equally long ones.
struct CfPieces {
  int32_t ntasks = 0;
  int32_t most = 0;
  int64_t npieces = 0;
  char* slab = nullptr;        // one allocation that holds the arrays below
  int4* recs = nullptr;        // [ntasks x pieces per task] (first rating, its high
                               // word, ratings, vertex); unused: 0 ratings
  int32_t* slots = nullptr;    // [npieces] a vertex's pieces' slots, in rating order
  int64_t* poff = nullptr;     // [n+1] first piece of each vertex
  int32_t* many = nullptr;     // [most_many + 2] a list of vertices with many pieces (cf.cu)
  int32_t most_many = 0;
  float* gpart = nullptr;      // [slots][K] piece gradients
  int64_t bytes = 0;
};

// Lay out one side: n vertices with R ratings, K dimensions; room for a list of
// vertices that have more than `few` pieces.  Synchronizes.
int cf_pieces_build(CfPieces* c, int64_t n, int64_t R, int K, const int64_t* off, int few,
                    cudaStream_t s);
void cf_pieces_free(CfPieces* c);

// Piece gradients of one side into c.gpart; with_sse (side 0): the squared
// errors' sum.  self / other: the two sides' factors in their storage (nn
// neighbour rows).
int cf_rows_gather(const CfPieces& c, int K, bool bf16, int64_t nn, const int32_t* nbr,
                   const uint8_t* rate, const void* self, const void* other, bool with_sse,
                   double* partials, unsigned* counter, double* sse, int grid, cudaStream_t s);
int cf_rows_grid(int K, int* grid);  // blocks of a gather (partials: one each)

}  // namespace cg
