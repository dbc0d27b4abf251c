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
// time first).  Nothing waits on another block.
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
  int32_t vmax = 0;
  SegPlan plan;               // the graphs as staged segments: tasks, stream, carries
  int64_t* vbase = nullptr;   // [G+1] first vertex of each graph (from v0 on)
  int32_t* order = nullptr;   // [G] graphs by edge count, descending
  int32_t* ndang = nullptr;   // [G]
  int32_t* xbase = nullptr;   // [G+1] first carry of each graph
  int32_t* row_ptr = nullptr; // [rows+1] first edge of each non-empty row
  int32_t* idx = nullptr;     // [rows] local destination of each non-empty row
  float* inv = nullptr;       // [V]
  float* sums = nullptr;      // [V] row sums of graphs too large to keep them on chip
  unsigned* counter = nullptr;
  int64_t bytes = 0;
};

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

// The edge offsets at the graphs' first vertices.
__global__ void batch_ebase_kernel(const int64_t* __restrict__ offsets,
                                   const int64_t* __restrict__ vbase, int G,
                                   int64_t* __restrict__ ebase) {
  for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g <= G;
       g += (int64_t)gridDim.x * blockDim.x)
    ebase[g] = offsets[vbase[g]];
}

// (Offsets, sources and bases below are those of a part: vertices and edges are
// counted from its first ones, offsets from its first edge, e0, on.)
__global__ void batch_degree_kernel(const int32_t* __restrict__ src, const int64_t* __restrict__ ebase,
                                    const int64_t* __restrict__ vbase, int G, int64_t E,
                                    int32_t* __restrict__ outdeg) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    int lo = 0, hi = G + 1;  // graph of edge e: last g with ebase[g] <= e
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (ebase[mid] <= e) lo = mid + 1; else hi = mid;
    }
    const int g = lo - 1;
    const int32_t u = src[e];
    if (u >= 0 && (int64_t)u < vbase[g + 1] - vbase[g]) atomicAdd(outdeg + vbase[g] + u, 1);
  }
}

__global__ void batch_inv_kernel(const int32_t* __restrict__ outdeg, int64_t V,
                                 float* __restrict__ inv, const int64_t* __restrict__ offsets,
                                 int32_t* __restrict__ nonempty, int32_t* __restrict__ bad) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    inv[v] = outdeg[v] > 0 ? 1.0f / (float)outdeg[v] : 0.0f;
    nonempty[v] = offsets[v + 1] > offsets[v] ? 1 : 0;
    if (offsets[v + 1] < offsets[v]) atomicExch(bad, 1);
  }
}

// Non-empty rows (in vertex order): their starts and local destinations, and
// their sources in the plan's padded layout.
__global__ void batch_rows_kernel(const int64_t* __restrict__ offsets,
                                  const int32_t* __restrict__ src,
                                  const int64_t* __restrict__ rowpos,  // exclusive scan of nonempty
                                  const int64_t* __restrict__ vbase,
                                  const int64_t* __restrict__ ebase,
                                  const int64_t* __restrict__ cstart, int G, int64_t V, int64_t e0,
                                  int pad,
                                  uint32_t* __restrict__ colf, int32_t* __restrict__ row_ptr,
                                  int32_t* __restrict__ idx) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < V; v += nw) {
    const int64_t lo = offsets[v] - e0, hi = offsets[v + 1] - e0;
    if (hi <= lo) continue;
    int a = 0, b = G + 1;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if (vbase[mid] <= v) a = mid + 1; else b = mid;
    }
    const int g = a - 1;
    const int32_t n = (int32_t)(vbase[g + 1] - vbase[g]);
    if (lane == 0) {
      idx[rowpos[v]] = (int32_t)(v - vbase[g]);
      row_ptr[rowpos[v]] = (int32_t)lo;
    }
    const int64_t shift = cstart[g] - ebase[g];
    for (int64_t e = lo + lane; e < hi; e += 32) {
      const int32_t u = src[e];  // a source outside its graph contributes nothing
      colf[e + shift] = (uint32_t)u < (uint32_t)n ? (uint32_t)u : (uint32_t)pad;
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
  float* rank;     // [V] result (and the previous iterate where residuals are asked for)
  double* resid;   // [G * iters] or NULL
  unsigned* counter;
  int G;
  int iters;
  int room;        // floats of dynamic shared memory behind the contrib vector
  float d;
};

template <int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
batch_pagerank_kernel(BatchArgs a) {
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
      const unsigned q = atomicAdd(a.counter, 1u);
      s_g = (int)q < a.G ? a.order[q] : -1;
    }
    __syncthreads();
    const int g = s_g;
    if (g < 0) break;
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
  cudaFree(b->vbase);
  cudaFree(b->order);
  cudaFree(b->ndang);
  cudaFree(b->xbase);
  cudaFree(b->row_ptr);
  cudaFree(b->idx);
  cudaFree(b->inv);
  cudaFree(b->sums);
  cudaFree(b->counter);
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

// Lays out one part (its G, g0, v0, e0, V, E and vmax are set); vbase and ebase:
// its graphs' first vertices and edges, counted from its own first ones.
int build_part(BatchPart* b, const std::vector<int64_t>& vbase, const std::vector<int64_t>& ebase,
               const int64_t* offsets, const int32_t* src, cudaStream_t s) {
  const int G = b->G;
  std::vector<int32_t> order(G);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int x, int y) {
    return ebase[x + 1] - ebase[x] > ebase[y + 1] - ebase[y];
  });
  const int64_t V = b->V, E = b->E;
  CG_TRY(seg_plan_alloc(E, G, ebase, vbase, &b->plan, s));
  SegPlan* p = &b->plan;
  const int64_t* d_ebase = p->meta + (G + 1);
  const int64_t* cstart = p->meta + 2 * (G + 1);
  CG_CUDA(cudaMalloc((void**)&b->vbase, sizeof(int64_t) * (G + 1)));
  CG_CUDA(cudaMalloc((void**)&b->order, sizeof(int32_t) * G));
  CG_CUDA(cudaMalloc((void**)&b->ndang, sizeof(int32_t) * G));
  CG_CUDA(cudaMalloc((void**)&b->xbase, sizeof(int32_t) * (G + 1)));
  CG_CUDA(cudaMalloc((void**)&b->inv, sizeof(float) * (size_t)V));
  CG_CUDA(cudaMalloc((void**)&b->sums, sizeof(float) * (size_t)V));
  CG_CUDA(cudaMalloc((void**)&b->counter, sizeof(unsigned)));
  CG_CUDA(cudaMemcpyAsync(b->vbase, vbase.data(), sizeof(int64_t) * (G + 1),
                          cudaMemcpyHostToDevice, s));
  CG_CUDA(cudaMemcpyAsync(b->order, order.data(), sizeof(int32_t) * G, cudaMemcpyHostToDevice, s));
  // scratch: out-degree, non-empty flags and their scan
  Scratch tmp(s, 2 * Scratch::round(4 * (size_t)V) + Scratch::round(8 * (size_t)(V + 1)) +
                     scan_scratch(V) + 256);
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
  batch_inv_kernel<<<grid_for(V, 256), 256, 0, s>>>(outdeg, V, b->inv, offsets, nonempty, bad);
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
  CG_CUDA(cudaMalloc((void**)&b->idx, sizeof(int32_t) * (size_t)(b->rows + 1)));
  CG_CUDA(cudaMalloc((void**)&b->row_ptr, sizeof(int32_t) * (size_t)(b->rows + 1)));
  const int32_t end = (int32_t)E;
  CG_CUDA(cudaMemcpyAsync(b->row_ptr + b->rows, &end, sizeof(int32_t), cudaMemcpyHostToDevice, s));
  batch_rows_kernel<<<grid_for(V * 32, 256, 16), 256, 0, s>>>(
      offsets, src, rowpos, b->vbase, d_ebase, cstart, G, V, b->e0, batch_pad(*b), p->colf,
      b->row_ptr, b->idx);
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
  b->bytes = seg_plan_bytes(*p) + 8 * V + 8 * (b->rows + 1) + 20 * (int64_t)(G + 1);
  return CG_OK;
}

int build_batch(cg_batch* b, const int64_t* vbase, const int64_t* offsets, const int32_t* src,
                cudaStream_t s) {
  const int G = b->G;
  std::vector<int64_t> ebase(G + 1, 0);
  {
    Scratch tmp(s, 2 * Scratch::round(8 * (size_t)(G + 1)));
    int64_t *d_v = nullptr, *d_e = nullptr;
    CG_CUDA(tmp.get(&d_v, G + 1));
    CG_CUDA(tmp.get(&d_e, G + 1));
    CG_CUDA(cudaMemcpyAsync(d_v, vbase, sizeof(int64_t) * (G + 1), cudaMemcpyHostToDevice, s));
    batch_ebase_kernel<<<grid_for(G + 1, 256), 256, 0, s>>>(offsets, d_v, G, d_e);
    CG_LAUNCH_CHECK();
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
      if (q > 0) p.vmax = std::max(p.vmax, (int32_t)(vb[q] - vb[q - 1]));
    }
    CG_TRY(build_part(&p, vb, eb, offsets + p.v0, src + p.e0, s));
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
  const size_t smem = std::max(least, std::min(2 * least, most));
  BatchArgs a;
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
  a.rank = rank + b.v0;
  a.resid = resid ? resid + b.g0 * iterations : nullptr;
  a.counter = b.counter;
  a.G = b.G;
  a.iters = iterations;
  a.room = (int)((smem - least) / sizeof(float));
  a.d = (float)damping;
  const int per_sm = std::max(1, std::min(1024 / threads,
                                          (int)(232448 / std::max<size_t>(smem + 2048, 1))));
  const int grid = std::min<int>(b.G, di.sm_count * per_sm);
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
