// Batched PageRank over many small graphs in one persistent launch.
//
// Each graph is small enough that its whole contrib vector fits in one SM's
// shared memory, so a graph is its own single shared-memory segment (k = 1
// in the paper's terms) and a block runs all of its iterations on chip:
//   gather   the staged segments' warp tasks (staged_stream.cuh: rows of one
//            length class, 16-bit sources) fold contrib from shared memory and
//            write each row's sum to its destination's place in a dense
//            vector, kept in shared memory where both fit; destinations
//            without in-edges keep their 0;
//   update   the normalised vertex update, the FP64 dangling mass and the L1
//            residual, and the next contrib written back into shared memory.
// Rows longer than one task (4096 edges) are completed in between.  Ranks are
// written by the last iteration alone unless residuals are asked for.
// Graphs are handed out largest first through an atomic counter, so the
// biggest ones start first and small ones fill in behind (longest processing
// time first).  Nothing waits on another block.  Tiny graphs that come in thousands
// are handed out last, to a warp each, and have plain rows (kTinyGraphs below).
//
// The earlier kernel walked 256-edge chunks of 32-bit flagged sources with a
// scan per chunk, stored the row sums in row order, scattered them into the
// contrib vector's place, and read and wrote the ranks every iteration, with
// seven barriers.  1,024 graphs of scales 8-15, 20 iterations: 5.17 -> 2.13 ms;
// 40 graphs of scales 8-12 (one block each, the largest decides): 402 -> 151 us.
#include <algorithm>
#include <numeric>
#include <vector>

#include "staged_stream.cuh"

namespace cg {

// Consecutive graphs that are laid out and launched together.
struct BatchPart {
  int32_t G = 0;
  int64_t g0 = 0, v0 = 0, e0 = 0;  // first graph, vertex and edge
  int64_t V = 0, E = 0, rows = 0;
  int32_t nstaged = 0;        // graphs that are not tiny
  int32_t vmax = 0, tmax = 0; // vertices of the largest of them and of the largest tiny one
  SegPlan plan;               // the graphs as staged segments: tasks, stream, carries
  char* slab = nullptr;       // one allocation that holds the arrays up to sums
  int64_t* vbase = nullptr;   // [G+1] first vertex of each graph (from v0 on)
  int32_t* order = nullptr;   // [G] graphs by edge count, descending, the tiny ones last
  int32_t* ndang = nullptr;   // [G]
  int32_t* xbase = nullptr;   // [G+1] first carry of each graph
  unsigned* counter = nullptr;
  float* inv = nullptr;       // [V]
  float* sums = nullptr;      // [V] row sums of graphs too large to keep them on chip
  int32_t* row_ptr = nullptr; // [rows+1] first edge of each non-empty row
  int32_t* idx = nullptr;     // [rows] local destination of each, in the same allocation
  longlong2* tiny = nullptr;  // [G] a tiny graph's first source and row start, (-1, -) for
                              // the others; NULL where there is no tiny one
  uint16_t* trow = nullptr;   // where the tiny graphs' rows begin among their sources (one
                              // entry more than rows), and these; same allocation as tiny
  uint8_t* tcol = nullptr;
  int64_t bytes = 0;
};

// Tiny graphs, where there are thousands, have plain rows in place of staged
// tasks, which take 0.6 to 2 KB for every length class that a graph's rows meet
// (kept for 20,000 graphs of 25 vertices and 50 edges: 134 MB so, 10 MB with plain
// rows), and a warp each in place of a block.  Up to the limits below no batch of
// 4,096 and more was slower than with a block each, at 256 threads per block,
// where blocks are fastest (4.66 ms at 1024 threads and 1.19 at 256 for those
// 20,000, 0.28 and 0.26 so; 12,000 of 64 vertices and 1,024 edges 0.54 of the
// time; 7,800 of 64 and 1,536: 0.96).  One graph on its own takes up to three
// times as long on a warp, hence only from kTinyGraphs on.
constexpr int kTinyVertices = 255;
constexpr int kTinyEdges = 1280;
constexpr int kTinyRow = 255;  // edges of the longest row
constexpr int kTinyGraphs = 4096;
constexpr uint8_t kOutside = 255;  // a source outside its graph

// A part ends before it has more than this many graphs, vertices or edges (a
// graph of more edges has one to itself): its places then fit 32 bits, and the
// scratch of its build, 4 KB per graph, stays below 1 GB.  A batch within one part
// is one launch.
constexpr int64_t kPartGraphs = (int64_t)1 << 18;
constexpr int64_t kPartVertices = (int64_t)1 << 30;
constexpr int64_t kPartEdges = (int64_t)1 << 30;

}  // namespace cg

struct cg_batch {
  int device = 0;
  int32_t G = 0;
  std::vector<cg::BatchPart> parts;
  int threads = 1024;
  int64_t bytes = 0;
};

namespace cg {
namespace {

// The edge offsets at the graphs' first vertices, and whether a graph is tiny:
// a warp per graph.
__global__ void batch_look_kernel(const int64_t* __restrict__ offsets,
                                  const int64_t* __restrict__ vbase, int G,
                                  int64_t* __restrict__ ebase, uint8_t* __restrict__ tiny) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t g = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; g <= G; g += nw) {
    const int64_t v0 = vbase[g], v1 = g < G ? vbase[g + 1] : v0;
    if (lane == 0) ebase[g] = offsets[v0];
    if (g == G) break;
    bool fits = v1 - v0 <= kTinyVertices;
    if (fits) fits = offsets[v1] - offsets[v0] <= kTinyEdges;
    if (fits)
      for (int64_t v = v0 + lane; v < v1; v += 32) {
        const int64_t n = offsets[v + 1] - offsets[v];
        fits = fits && n >= 0 && n <= kTinyRow;
      }
    fits = __all_sync(0xffffffffu, fits);
    if (lane == 0) tiny[g] = fits;
  }
}

// The graph that vertex v lies in: the last g with vbase[g] <= v.
__device__ __forceinline__ int graph_of(const int64_t* __restrict__ vbase, int G, int64_t v) {
  int lo = 0, hi = G + 1;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (vbase[mid] <= v) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

// (Offsets, sources and bases below are those of a part: vertices and edges are
// counted from its first ones, offsets from its first edge, e0, on.)
__global__ void batch_degree_kernel(const int32_t* __restrict__ src, const int64_t* __restrict__ ebase,
                                    const int64_t* __restrict__ vbase, int G, int64_t E,
                                    int32_t* __restrict__ outdeg) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int g = graph_of(ebase, G, e);
    const int32_t u = src[e];
    if (u >= 0 && (int64_t)u < vbase[g + 1] - vbase[g]) atomicAdd(outdeg + vbase[g] + u, 1);
  }
}

// (nonempty: of the rows that become staged ones)
__global__ void batch_inv_kernel(const int32_t* __restrict__ outdeg, int64_t V,
                                 float* __restrict__ inv, const int64_t* __restrict__ offsets,
                                 const int64_t* __restrict__ vbase, int G,
                                 const longlong2* __restrict__ tiny,
                                 int32_t* __restrict__ nonempty, int32_t* __restrict__ bad) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    inv[v] = outdeg[v] > 0 ? 1.0f / (float)outdeg[v] : 0.0f;
    bool staged = offsets[v + 1] > offsets[v];
    if (staged && tiny) staged = tiny[graph_of(vbase, G, v)].x < 0;
    nonempty[v] = staged ? 1 : 0;
    if (offsets[v + 1] < offsets[v]) atomicExch(bad, 1);
  }
}

// Non-empty rows (in vertex order): their starts and local destinations, and
// their sources in the plan's padded layout; the tiny graphs' rows.  sbase: the
// graphs' first edges among the staged ones.
struct RowsOut {
  uint32_t* colf;
  int32_t* row_ptr;
  int32_t* idx;
  const longlong2* tiny;
  uint16_t* trow;
  uint8_t* tcol;
};
__global__ void batch_rows_kernel(const int64_t* __restrict__ offsets,
                                  const int32_t* __restrict__ src,
                                  const int64_t* __restrict__ rowpos,  // exclusive scan of nonempty
                                  const int64_t* __restrict__ vbase,
                                  const int64_t* __restrict__ ebase,
                                  const int64_t* __restrict__ sbase,
                                  const int64_t* __restrict__ cstart, int G, int64_t V, int64_t e0,
                                  int pad, RowsOut out) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < V; v += nw) {
    const int64_t lo = offsets[v] - e0, hi = offsets[v + 1] - e0;
    if (hi <= lo && !out.tiny) continue;
    const int g = graph_of(vbase, G, v);
    const int32_t n = (int32_t)(vbase[g + 1] - vbase[g]);
    const int64_t eb = ebase[g];
    const longlong2 t = out.tiny ? out.tiny[g] : make_longlong2(-1, 0);
    if (t.x >= 0) {
      uint16_t* row = out.trow + t.y + (v - vbase[g]);
      if (lane == 0) {
        row[0] = (uint16_t)(lo - eb);
        if (v + 1 == vbase[g + 1]) row[1] = (uint16_t)(hi - eb);
      }
    } else if (lane == 0 && hi > lo) {
      out.idx[rowpos[v]] = (int32_t)(v - vbase[g]);
      out.row_ptr[rowpos[v]] = (int32_t)(lo - eb + sbase[g]);
    }
    for (int64_t e = lo + lane; e < hi; e += 32) {
      const int32_t u = src[e];  // a source outside its graph contributes nothing
      const bool inside = (uint32_t)u < (uint32_t)n;
      if (t.x >= 0)
        out.tcol[t.x + (e - eb)] = inside ? (uint8_t)u : kOutside;
      else
        out.colf[cstart[g] + (e - eb)] = inside ? (uint32_t)u : (uint32_t)pad;
    }
  }
}

// First carry of each graph: carries lie in row order.
__global__ void batch_xbase_kernel(const int32_t* __restrict__ xrow, int64_t nx,
                                   const int64_t* __restrict__ row_base, int G,
                                   int32_t* __restrict__ xbase) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g <= G; g += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = nx;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (xrow[mid] < row_base[g]) lo = mid + 1; else hi = mid;
    }
    xbase[g] = (int32_t)lo;
  }
}

__global__ void batch_dangling_kernel(const int32_t* __restrict__ outdeg,
                                      const int64_t* __restrict__ vbase, int G,
                                      int32_t* __restrict__ ndang) {
  for (int g = blockIdx.x; g < G; g += gridDim.x) {
    int c = 0;
    for (int64_t v = vbase[g] + threadIdx.x; v < vbase[g + 1]; v += blockDim.x)
      c += outdeg[v] == 0;
    c = warp_sum(c);
    __shared__ int sh[32];
    if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = c;
    __syncthreads();
    if (threadIdx.x == 0) {
      int t = 0;
      for (int q = 0; q < (int)(blockDim.x >> 5); ++q) t += sh[q];
      ndang[g] = t;
    }
    __syncthreads();
  }
}

struct BatchArgs {
  StagedTasks tasks;
  const int32_t* idx;
  const int32_t* xbase;
  const int32_t* xrow;
  float* carry;
  const float* inv;
  const int64_t* vbase;
  const int32_t* order;
  const int32_t* ndang;
  float* sums;
  const longlong2* tiny;
  const uint16_t* trow;
  const uint8_t* tcol;
  float* rank;     // [V] result (and the previous iterate where residuals are asked for)
  double* resid;   // [G * iters] or NULL
  unsigned* counter;
  int G;
  int nstaged;     // graphs that a block solves; behind them in `order` the tiny ones,
  int bundle;      // so many of which a block's warps take at once, one each
  int stride;      // floats of a tiny graph's vector (a warp has it and its row sums)
  int iters;
  int room;        // floats of dynamic shared memory behind the contrib vector
  float d;
};

// x at source e of a row of n, 0 behind its end and where the source is outside.
__device__ __forceinline__ float tiny_at(const uint8_t* __restrict__ col, int e, int n,
                                         const float* x) {
  const int u = e < n ? __ldg(col + e) : kOutside;
  return u != kOutside ? x[u] : 0.0f;
}

// The row sums of vertices v0 .. v0 + 31 (v: this lane's, with n sources from col
// on), each in the order in which a staged task adds it: up to 8 sources one after
// the other; up to 16 the even and the odd ones apart, a lane per row; up to 16
// 2^lg so on each of 2^lg lanes (here four, with up to four of those lanes' parts
// each, for eight rows at a time), then a tree over the lanes.
__device__ __forceinline__ void tiny_rows(const uint8_t* __restrict__ col, int lo, int n, int v,
                                          int v0, const float* x, float* sums) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31, sub = lane & 3, grp = lane >> 2;
  if (n <= 16) {
    float a = 0.0f, b = 0.0f;
    for (int e = 0; e < n; e += 4) {
      const uint8_t* c = col + lo;
      const float w[4] = {tiny_at(c, e, n, x), tiny_at(c, e + 1, n, x), tiny_at(c, e + 2, n, x),
                          tiny_at(c, e + 3, n, x)};
      if (n <= 8) {
        a += w[0]; a += w[1]; a += w[2]; a += w[3];
      } else {
        a += w[0]; b += w[1]; a += w[2]; b += w[3];
      }
    }
    if (v >= 0) sums[v] = a + b;
  }
  for (unsigned rest = __ballot_sync(kFull, n > 16); rest;) {
    unsigned t = rest;  // the group takes the grp-th row of the rest
    for (int q = 0; q < grp; ++q) t &= t - 1;
    const int at = t ? __ffs(t) - 1 : 0;
    const uint8_t* c = col + __shfl_sync(kFull, lo, at);
    const int len = __shfl_sync(kFull, n, at), m = t ? len : 0;
    const int lg = m <= 16 ? 0 : 28 - __clz(m - 1);  // m <= 16 << lg
    float w[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int l = sub + 4 * k;
      if (l >= 1 << lg) break;
      float a = 0.0f, b = 0.0f;
      for (int e = l; e < m; e += 4 << lg) {
        const float y[4] = {tiny_at(c, e, m, x), tiny_at(c, e + (1 << lg), m, x),
                            tiny_at(c, e + (2 << lg), m, x), tiny_at(c, e + (3 << lg), m, x)};
        a += y[0]; b += y[1]; a += y[2]; b += y[3];
      }
      w[k] = a + b;
    }
    __syncwarp();
    const int parts = __any_sync(kFull, m > 64) ? 4 : 1;  // (the other parts are 0)
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= parts) break;
      w[k] += __shfl_xor_sync(kFull, w[k], 1);
      w[k] += __shfl_xor_sync(kFull, w[k], 2);
    }
    if (sub == 0 && t) sums[v0 + at] = (w[0] + w[1]) + (w[2] + w[3]);
    for (int q = 0; q < 8; ++q) rest &= rest - 1;
  }
}

// All iterations of tiny graph g on one warp; x: contrib, and a.stride floats
// behind it the row sums.  Every sum is taken in the order of the block's way (a
// graph's ranks do not depend on the batch it is in).  Not inlined: the staged
// graphs' code keeps its registers.
__device__ __noinline__ void tiny_solve(const BatchArgs& a, int g, float* x) {
  constexpr unsigned kFull = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  const int64_t vb = a.vbase[g];
  const int V = (int)(a.vbase[g + 1] - vb);
  const longlong2 first = a.tiny[g];
  const uint16_t* row = a.trow + first.y;
  const uint8_t* col = a.tcol + first.x;
  const float* inv = a.inv + vb;
  float* rank = a.rank + vb;
  float* sums = x + a.stride;
  const bool residuals = a.resid != nullptr;
  const float base = (1.0f - a.d) / (float)V, r0 = 1.0f / (float)V;
  const double invV = 1.0 / (double)V;
  __syncwarp();  // the warp's previous graph is done with the vectors
  for (int v = lane; v < V; v += 32) {
    if (residuals) rank[v] = r0;
    x[v] = r0 * __ldg(inv + v);
  }
  double D = (double)a.ndang[g] * (double)r0;
  __syncwarp();
  for (int it = 0; it < a.iters; ++it) {
    const bool write = residuals || it == a.iters - 1;
    for (int v0 = 0; v0 < V; v0 += 32) {
      const int v = v0 + lane < V ? v0 + lane : -1;
      const int lo = v >= 0 ? __ldg(row + v) : 0, hi = v >= 0 ? __ldg(row + v + 1) : 0;
      tiny_rows(col, lo, hi - lo, v, v0, x, sums);
    }
    __syncwarp();
    const float Dv = (float)(D * invV);
    double dd = 0.0, rr = 0.0;  // lane c: those of vertices 32 c .. 32 c + 31, summed in FP32
    for (int c = 0; 32 * c < V; ++c) {
      const int v = 32 * c + lane;
      float dpart = 0.0f, rpart = 0.0f;
      if (v < V) {
        const float iv = __ldg(inv + v);
        const float r = base + a.d * (sums[v] + Dv);
        if (residuals) rpart = fabsf(r - rank[v]);
        if (write) rank[v] = r;
        x[v] = r * iv;
        if (iv == 0.0f) dpart = r;
      }
      const float d = __shfl_sync(kFull, warp_sum(dpart), 0);
      if (lane == c) dd = (double)d;
      if (residuals) {
        const float q = __shfl_sync(kFull, warp_sum(rpart), 0);
        if (lane == c) rr = (double)q;
      }
    }
    D = __shfl_sync(kFull, warp_sum(dd), 0);
    if (residuals) {
      rr = warp_sum(rr);
      if (lane == 0) a.resid[(int64_t)g * a.iters + it] = rr;
    }
    __syncwarp();
  }
}

template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
batch_pagerank_kernel(const __grid_constant__ BatchArgs a) {
  constexpr int WARPS = THREADS / 32;
  extern __shared__ __align__(16) float xs[];  // contrib, the identity, then the row sums
  __shared__ int s_g;
  __shared__ double s_red[2][WARPS];
  __shared__ double s_D;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const bool residuals = a.resid != nullptr;
  if (tid == 0) xs[a.tasks.pad] = 0.0f;
  for (;;) {
    __syncthreads();
    if (tid == 0) {
      const int q = (int)atomicAdd(a.counter, 1u);
      const int64_t t = a.nstaged + (int64_t)(q - a.nstaged) * a.bundle;  // first of a bundle
      s_g = q < a.nstaged ? a.order[q] : t < a.G ? -1 - (int)t : INT32_MIN;
    }
    __syncthreads();
    const int g = s_g;
    if (g < 0) {
      if (g == INT32_MIN) break;
      const int t = -1 - g + w;  // (staged graphs are all handed out before)
      if (w < a.bundle && t < a.G) tiny_solve(a, a.order[t], xs + w * 2 * a.stride);
      continue;
    }
    const int64_t vb = a.vbase[g];
    const int V = (int)(a.vbase[g + 1] - vb);
    const int32_t t0 = a.tasks.seg_task[g], t1 = a.tasks.seg_task[g + 1];
    const int32_t x0 = a.xbase[g], x1 = a.xbase[g + 1];
    const float base = (1.0f - a.d) / (float)V;
    const double invV = 1.0 / (double)V;
    float* rank = a.rank + vb;
    const float* inv = a.inv + vb;
    float* sums = V <= a.room ? xs + a.tasks.pad + 4 : a.sums + vb;
    // r_0 = 1/V
    const float r0 = 1.0f / (float)V;
    for (int v = tid; v < V; v += THREADS) {
      if (residuals) rank[v] = r0;
      xs[v] = r0 * inv[v];
      sums[v] = 0.0f;
    }
    double D = (double)a.ndang[g] * (double)r0;
    __syncthreads();
    for (int it = 0; it < a.iters; ++it) {
      const bool write = residuals || it == a.iters - 1;
      staged_run<SumF32>(a.tasks, t0, t1, w, WARPS, xs, sums, a.carry);
      __syncthreads();
      if (x1 > x0) {  // rows of more than 4096 edges: the first full piece's thread sums them
        for (int x = x0 + tid; x < x1; x += THREADS) {
          const int32_t r = a.xrow[x];
          if (x > x0 && a.xrow[x - 1] == r) continue;
          float s = a.carry[x];
          for (int y = x + 1; y < x1 && a.xrow[y] == r; ++y) s += a.carry[y];
          sums[a.idx[r]] += s;
        }
        __syncthreads();
      }
      // vertex update, next contrib, FP64 dangling mass and residual
      const float Dv = (float)(D * invV);
      float dpart = 0.0f, rpart = 0.0f;
      constexpr int U = 8;  // vertices per thread whose inputs are loaded together
      for (int v0 = tid; v0 < V; v0 += THREADS * U) {
        float iv[U], sm[U], old[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const int v = v0 + u * THREADS;
          iv[u] = v < V ? __ldg(inv + v) : 0.0f;
          sm[u] = v < V ? sums[v] : 0.0f;
          old[u] = residuals && v < V ? rank[v] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {  // the same vertex order as one at a time
          const int v = v0 + u * THREADS;
          if (v < V) {
            const float r = base + a.d * (sm[u] + Dv);
            if (residuals) rpart += fabsf(r - old[u]);
            if (write) rank[v] = r;
            xs[v] = r * iv[u];
            if (iv[u] == 0.0f) dpart += r;
          }
        }
      }
      // the lanes' partials in FP32 over groups of 2o lanes while a group
      // holds at most 256 ranks (ceil(V / THREADS) per lane), then in FP64
      const int per_lane = (V + THREADS - 1) / THREADS;
      int o = 16;
      while (o >= 1 && 2 * o * per_lane > 256) o >>= 1;
      for (int f = o; f >= 1; f >>= 1) {
        dpart += __shfl_down_sync(0xffffffffu, dpart, f);
        if (residuals) rpart += __shfl_down_sync(0xffffffffu, rpart, f);
      }
      double dd = (double)dpart, rr = (double)rpart;
      for (int f = 16; f > o; f >>= 1) {
        dd += __shfl_down_sync(0xffffffffu, dd, f);
        if (residuals) rr += __shfl_down_sync(0xffffffffu, rr, f);
      }
      if (lane == 0) {
        s_red[0][w] = dd;
        s_red[1][w] = rr;
      }
      __syncthreads();
      // the warps' sums, added by one warp in a fixed tree (FP64 runs at a
      // small fraction of the FP32 rate on this GPU)
      if (w == 0) {
        const double Dn = warp_sum(lane < WARPS ? s_red[0][lane] : 0.0);
        if (lane == 0) s_D = Dn;
      } else if (residuals && w == 1) {
        const double Rn = warp_sum(lane < WARPS ? s_red[1][lane] : 0.0);
        if (lane == 0) a.resid[(int64_t)g * a.iters + it] = Rn;
      }
      __syncthreads();
      D = s_D;
    }
  }
}

void free_part(BatchPart* b) {
  seg_plan_free(&b->plan);
  cudaFree(b->slab);
  cudaFree(b->row_ptr);
  cudaFree(b->tiny);
}

void free_batch(cg_batch* b) {
  for (BatchPart& p : b->parts) free_part(&p);
}

// row_base[g] = first non-empty row of graph g.
__global__ void batch_row_base_kernel(const int64_t* __restrict__ rowpos,
                                      const int64_t* __restrict__ vbase, int G,
                                      int64_t* __restrict__ row_base) {
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g <= G; g += gridDim.x * blockDim.x)
    row_base[g] = rowpos[vbase[g]];
}

// the entry behind the largest contrib vector that holds the sum's identity
int batch_pad(const BatchPart& b) { return (b.vmax + 3) & ~3; }

// Lays out one part (its G, g0, v0, e0, V and E are set); vbase and ebase:
// its graphs' first vertices and edges, counted from its own first ones.
int build_part(BatchPart* b, const std::vector<int64_t>& vbase, const std::vector<int64_t>& ebase,
               std::vector<uint8_t> is_tiny, const int64_t* offsets, const int32_t* src,
               cudaStream_t s) {
  const int G = b->G;
  if (std::count(is_tiny.begin(), is_tiny.end(), 1) < kTinyGraphs)
    std::fill(is_tiny.begin(), is_tiny.end(), 0);
  // the staged graphs' edges, and the tiny graphs' places
  std::vector<int64_t> sbase(G + 1, 0);
  std::vector<longlong2> tiny(G, make_longlong2(-1, 0));
  int64_t ncol = 0, nrow = 0;
  for (int g = 0; g < G; ++g) {
    const int64_t n = ebase[g + 1] - ebase[g];
    sbase[g + 1] = sbase[g] + (is_tiny[g] ? 0 : n);
    const int32_t vertices = (int32_t)(vbase[g + 1] - vbase[g]);
    if (!is_tiny[g]) {
      ++b->nstaged;
      b->vmax = std::max(b->vmax, vertices);
    } else {
      b->tmax = std::max(b->tmax, vertices);
      tiny[g] = make_longlong2(ncol, nrow);
      ncol += n;
      nrow += vbase[g + 1] - vbase[g] + 1;
    }
  }
  std::vector<int32_t> order(G);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    if (is_tiny[x] != is_tiny[y]) return is_tiny[x] < is_tiny[y];
    return ebase[x + 1] - ebase[x] > ebase[y + 1] - ebase[y];
  });
  const int64_t V = b->V, E = b->E;
  CG_TRY(seg_plan_alloc(sbase[G], G, sbase, vbase, &b->plan, s));
  SegPlan* p = &b->plan;
  const int64_t* d_sbase = p->meta + (G + 1);
  const int64_t* cstart = p->meta + 2 * (G + 1);
  const size_t g8 = Scratch::round(8 * (size_t)(G + 1)), g4 = Scratch::round(4 * (size_t)(G + 1)),
               v4 = Scratch::round(4 * (size_t)V);
  CG_CUDA(cudaMalloc((void**)&b->slab, g8 + 3 * g4 + 256 + 2 * v4));
  b->vbase = reinterpret_cast<int64_t*>(b->slab);
  b->order = reinterpret_cast<int32_t*>(b->slab + g8);
  b->ndang = reinterpret_cast<int32_t*>(b->slab + g8 + g4);
  b->xbase = reinterpret_cast<int32_t*>(b->slab + g8 + 2 * g4);
  b->counter = reinterpret_cast<unsigned*>(b->slab + g8 + 3 * g4);
  b->inv = reinterpret_cast<float*>(b->slab + g8 + 3 * g4 + 256);
  b->sums = reinterpret_cast<float*>(b->slab + g8 + 3 * g4 + 256 + v4);
  CG_CUDA(cudaMemcpyAsync(b->vbase, vbase.data(), sizeof(int64_t) * (G + 1),
                          cudaMemcpyHostToDevice, s));
  CG_CUDA(cudaMemcpyAsync(b->order, order.data(), sizeof(int32_t) * G, cudaMemcpyHostToDevice, s));
  const size_t tiny_bytes = nrow > 0 ? 16 * (size_t)G + 2 * (size_t)nrow + (size_t)ncol : 0;
  if (nrow > 0) {
    CG_CUDA(cudaMalloc((void**)&b->tiny, tiny_bytes));
    b->trow = reinterpret_cast<uint16_t*>(b->tiny + G);
    b->tcol = reinterpret_cast<uint8_t*>(b->trow + nrow);
    CG_CUDA(cudaMemcpyAsync(b->tiny, tiny.data(), sizeof(longlong2) * G, cudaMemcpyHostToDevice,
                            s));
  }
  // scratch: out-degree, non-empty flags and their scan, the graphs' first edges
  Scratch tmp(s, 2 * Scratch::round(4 * (size_t)V) + Scratch::round(8 * (size_t)(V + 1)) +
                     scan_scratch(V) + 256 + Scratch::round(8 * (size_t)(G + 1)));
  int64_t* d_ebase = nullptr;
  CG_CUDA(tmp.get(&d_ebase, G + 1));
  CG_CUDA(cudaMemcpyAsync(d_ebase, ebase.data(), sizeof(int64_t) * (G + 1),
                          cudaMemcpyHostToDevice, s));
  int32_t *outdeg = nullptr, *nonempty = nullptr;
  int64_t* rowpos = nullptr;
  int32_t* bad = nullptr;
  CG_CUDA(tmp.get(&outdeg, V));
  CG_CUDA(tmp.get(&nonempty, V));
  CG_CUDA(tmp.get(&rowpos, V + 1));
  CG_CUDA(tmp.get(&bad, 1));
  CG_CUDA(cudaMemsetAsync(bad, 0, sizeof(int32_t), s));
  CG_CUDA(cudaMemsetAsync(outdeg, 0, sizeof(int32_t) * (size_t)V, s));
  if (E > 0) {
    batch_degree_kernel<<<grid_for(E, 256), 256, 0, s>>>(src, d_ebase, b->vbase, G, E, outdeg);
    CG_LAUNCH_CHECK();
  }
  batch_inv_kernel<<<grid_for(V, 256), 256, 0, s>>>(outdeg, V, b->inv, offsets, b->vbase, G,
                                               b->tiny, nonempty, bad);
  CG_LAUNCH_CHECK();
  batch_dangling_kernel<<<std::min(G, 4096), 256, 0, s>>>(outdeg, b->vbase, G, b->ndang);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i32_to_i64(nonempty, rowpos, V, s, &tmp));
  batch_row_base_kernel<<<grid_for(G + 1, 256), 256, 0, s>>>(rowpos, b->vbase, G, p->meta);
  CG_LAUNCH_CHECK();
  std::vector<int64_t> rbase(G + 1, 0);
  CG_CUDA(cudaMemcpyAsync(rbase.data(), p->meta, sizeof(int64_t) * (G + 1),
                          cudaMemcpyDeviceToHost, s));
  int32_t hbad = 0;
  CG_CUDA(cudaMemcpyAsync(&hbad, bad, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  if (hbad) {
    set_error("pr_batch_create: offsets decrease within a graph");
    return CG_ERR_INVALID_ARG;
  }
  b->rows = rbase[G];
  CG_CUDA(cudaMalloc((void**)&b->row_ptr, sizeof(int32_t) * 2 * (size_t)(b->rows + 1)));
  b->idx = b->row_ptr + b->rows + 1;
  const int32_t end = (int32_t)sbase[G];
  CG_CUDA(cudaMemcpyAsync(b->row_ptr + b->rows, &end, sizeof(int32_t), cudaMemcpyHostToDevice, s));
  batch_rows_kernel<<<grid_for(V * 32, 256, 16), 256, 0, s>>>(
      offsets, src, rowpos, b->vbase, d_ebase, d_sbase, cstart, G, V, b->e0, batch_pad(*b),
      RowsOut{p->colf, b->row_ptr, b->idx, b->tiny, b->trow, b->tcol});
  CG_LAUNCH_CHECK();
  p->rows = b->rows;
  p->rp32 = b->row_ptr;
  p->row_base = rbase;
  CG_TRY(staged_build(p, G, batch_pad(*b), 0, s, b->idx));
  batch_xbase_kernel<<<grid_for(G + 1, 256), 256, 0, s>>>(p->carry_row, p->ncarry, p->meta, G,
                                                          b->xbase);
  CG_LAUNCH_CHECK();
  CG_CUDA(cudaStreamSynchronize(s));
  // the flagged 32-bit sources were only the stream's input
  cudaFree(p->colf);
  p->colf = nullptr;
  p->colf_len = 0;
  b->bytes = seg_plan_bytes(*p) + 8 * V + 8 * (b->rows + 1) + 20 * (int64_t)(G + 1) +
             (int64_t)tiny_bytes;
  return CG_OK;
}

int build_batch(cg_batch* b, const int64_t* vbase, const int64_t* offsets, const int32_t* src,
                cudaStream_t s) {
  const int G = b->G;
  std::vector<int64_t> ebase(G + 1, 0);
  std::vector<uint8_t> tiny(G, 0);
  {
    Scratch tmp(s, 2 * Scratch::round(8 * (size_t)(G + 1)) + Scratch::round((size_t)G));
    int64_t *d_v = nullptr, *d_e = nullptr;
    uint8_t* d_t = nullptr;
    CG_CUDA(tmp.get(&d_t, G));
    CG_CUDA(tmp.get(&d_v, G + 1));
    CG_CUDA(tmp.get(&d_e, G + 1));
    CG_CUDA(cudaMemcpyAsync(d_v, vbase, sizeof(int64_t) * (G + 1), cudaMemcpyHostToDevice, s));
    batch_look_kernel<<<grid_for(((int64_t)G + 1) * 32, 256), 256, 0, s>>>(offsets, d_v, G, d_e,
                                                                           d_t);
    CG_LAUNCH_CHECK();
    CG_CUDA(cudaMemcpyAsync(tiny.data(), d_t, (size_t)G, cudaMemcpyDeviceToHost, s));
    CG_CUDA(cudaMemcpyAsync(ebase.data(), d_e, sizeof(int64_t) * (G + 1), cudaMemcpyDeviceToHost,
                            s));
    CG_CUDA(cudaStreamSynchronize(s));
  }
  if (ebase[0] != 0) {
    set_error("pr_batch_create: offsets must start at 0");
    return CG_ERR_INVALID_ARG;
  }
  for (int g = 0; g < G; ++g) {
    if (ebase[g + 1] < ebase[g]) {
      set_error("pr_batch_create: offsets decrease across graph %d", g);
      return CG_ERR_INVALID_ARG;
    }
    if (ebase[g + 1] - ebase[g] >= 0x7FFFFFFFLL) {
      set_error("pr_batch_create: graph %d has 2^31 - 1 edges or more", g);
      return CG_ERR_UNSUPPORTED;
    }
  }
  for (int64_t g = 0; g < G;) {
    int64_t h = g + 1;
    while (h < G && h - g < kPartGraphs && vbase[h + 1] - vbase[g] <= kPartVertices &&
           ebase[h + 1] - ebase[g] <= kPartEdges)
      ++h;
    b->parts.emplace_back();
    BatchPart& p = b->parts.back();
    p.G = (int32_t)(h - g);
    p.g0 = g;
    p.v0 = vbase[g];
    p.e0 = ebase[g];
    p.V = vbase[h] - p.v0;
    p.E = ebase[h] - p.e0;
    std::vector<int64_t> vb(p.G + 1), eb(p.G + 1);
    for (int32_t q = 0; q <= p.G; ++q) {
      vb[q] = vbase[g + q] - p.v0;
      eb[q] = ebase[g + q] - p.e0;
    }
    CG_TRY(build_part(&p, vb, eb, {tiny.begin() + g, tiny.begin() + h}, offsets + p.v0, src + p.e0,
                      s));
    b->bytes += p.bytes;
    g = h;
  }
  return CG_OK;
}

int run_part(const BatchPart& b, int threads, int32_t iterations, double damping, float* rank,
             double* resid, cudaStream_t stream) {
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  // contrib, the identity and, behind them, row sums for as many vertices as fit,
  // up to the largest graph's
  const int pad = batch_pad(b);
  const size_t least = sizeof(float) * (size_t)(pad + 4);
  const size_t most = (size_t)(232448 - 2048);
  // (a tiny graph's contrib and row sums per warp)
  const int stride = (b.tmax + 3) & ~3, warps = threads / 32;
  const size_t smem = std::max({least, std::min(2 * least, most),
                                sizeof(float) * (size_t)(2 * stride * warps)});
  BatchArgs a{};
  a.tasks = StagedTasks{b.plan.cs, b.plan.desc, b.plan.seg_task, pad};
  a.idx = b.idx;
  a.xbase = b.xbase;
  a.xrow = b.plan.carry_row;
  a.carry = (float*)b.plan.carry;
  a.inv = b.inv;
  a.vbase = b.vbase;
  a.order = b.order;
  a.ndang = b.ndang;
  a.sums = b.sums;
  a.tiny = b.tiny;
  a.tcol = b.tcol;
  a.trow = b.trow;
  a.rank = rank + b.v0;
  a.resid = resid ? resid + b.g0 * iterations : nullptr;
  a.counter = b.counter;
  a.G = b.G;
  a.iters = iterations;
  a.room = (int)((smem - least) / sizeof(float));
  a.nstaged = b.nstaged;
  a.stride = stride;
  a.d = (float)damping;
  const int per_sm = std::max(1, std::min(1024 / threads,
                                          (int)(232448 / std::max<size_t>(smem + 2048, 1))));
  const int ntiny = b.G - b.nstaged, slots = di.sm_count * per_sm;
  a.bundle = std::max(1, std::min(warps, (int)ceil_div(ntiny, slots)));
  const int grid = std::min<int>(b.nstaged + (int)ceil_div(ntiny, a.bundle), slots);
  CG_CUDA(cudaMemsetAsync(b.counter, 0, sizeof(unsigned), stream));
  const void* fn = threads == 1024 ? (const void*)batch_pagerank_kernel<1024>
                   : threads == 512 ? (const void*)batch_pagerank_kernel<512>
                                    : (const void*)batch_pagerank_kernel<256>;
  if (smem > 48 * 1024)
    CG_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  if (threads == 1024)
    batch_pagerank_kernel<1024><<<grid, 1024, smem, stream>>>(a);
  else if (threads == 512)
    batch_pagerank_kernel<512><<<grid, 512, smem, stream>>>(a);
  else
    batch_pagerank_kernel<256><<<grid, 256, smem, stream>>>(a);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int pr_batch_create(int32_t G, const int64_t* host_vbase, const int64_t* offsets,
                    const int32_t* src, cg_batch** out, cudaStream_t stream) {
  CG_ARG(out != nullptr, "pr_batch_create: out is NULL");
  *out = nullptr;
  CG_ARG(G >= 1 && host_vbase && offsets, "pr_batch_create: bad arguments");
  CG_ARG(host_vbase[0] == 0, "pr_batch_create: vertex bases must start at 0");
  int32_t vmax = 0;
  for (int g = 0; g < G; ++g) {
    const int64_t n = host_vbase[g + 1] - host_vbase[g];
    CG_ARG(n >= 1, "pr_batch_create: graph %d has no vertex", g);
    CG_ARG(n <= 65536, "pr_batch_create: graph %d has %lld vertices (at most 65536: a graph's "
           "contrib must fit in shared memory)", g, (long long)n);
    vmax = std::max<int32_t>(vmax, (int32_t)n);
  }
  cg_batch* b = new cg_batch();
  CG_CUDA(cudaGetDevice(&b->device));
  b->G = G;
  const int cap = (int)((232448 - 2048) / 4);  // shared memory of one block, in floats
  if (vmax > cap) {
    delete b;
    set_error("pr_batch_create: largest graph (%d vertices) exceeds shared memory", vmax);
    return CG_ERR_UNSUPPORTED;
  }
  int st = build_batch(b, host_vbase, offsets, src, stream);
  if (st != CG_OK) {
    cudaStreamSynchronize(stream);
    free_batch(b);
    delete b;
    return st;
  }
  *out = b;
  return CG_OK;
}

int pr_batch_destroy(cg_batch* b) {
  if (!b) return CG_OK;
  int cur = 0;
  const int dev = b->device;
  cudaGetDevice(&cur);
  if (cur != dev) cudaSetDevice(dev);
  cudaDeviceSynchronize();
  free_batch(b);
  delete b;
  if (cur != dev) cudaSetDevice(cur);
  return CG_OK;
}

int pr_batch_set_threads(cg_batch* b, int32_t threads) {
  CG_ARG(b != nullptr, "pr_batch_set_threads: null handle");
  CG_ARG(threads == 256 || threads == 512 || threads == 1024,
         "pr_batch_set_threads: threads must be 256, 512 or 1024");
  b->threads = threads;
  return CG_OK;
}

int pr_batch_run(cg_batch* b, int32_t iterations, double damping, float* rank,
                 double* resid, cudaStream_t stream) {
  CG_ARG(b && rank, "pr_batch_run: null argument");
  CG_ARG(iterations >= 1, "pr_batch_run: iterations must be >= 1");
  CG_ARG(damping >= 0.0 && damping <= 1.0, "pr_batch_run: damping must be in [0, 1]");
  for (const BatchPart& p : b->parts)
    CG_TRY(run_part(p, b->threads, iterations, damping, rank, resid, stream));
  return CG_OK;
}

int pr_batched_graphs_run(cg_batch* b, int32_t iterations, double damping, float* rank,
                          double* resid, cudaStream_t stream) {
  return pr_batch_run(b, iterations, damping, rank, resid, stream);
}

}  // extern "C"
