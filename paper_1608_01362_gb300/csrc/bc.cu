// Betweenness centrality from a set of sources (the BC application of the
// paper's Table V, run from 12 sources), by Brandes' algorithm over
// frontiers: the activeness side of the EdgeMap / VertexSubset API of
// Section IV, on the clustered graph (Section V; for BC the paper credits its
// speed-up to the renumbering, the working set being too small for
// segmenting to pay).
//
// Forward phase, one BFS level at a time from the source (level 0, sigma 1):
//   push (small frontier: its out-edges): an unvisited w gets level L+1 by
//         compare-and-swap and joins the next frontier; every edge into a
//         level-(L+1) vertex adds sigma[u] to sigma[w] with an FP64 atomic;
//   pull (large frontier, bottom-up): the in-rows of the unvisited vertices are
//         summed over sigma of the frontier's vertices (a bit each); an
//         unvisited v whose sum is non-zero gets level L+1 and sigma = the sum.
// sigma counts shortest paths: integers, exact in FP64 in any order below
// 2^53, so levels and sigma do not depend on the direction or the order.
// Pull is taken when (frontier out-edges) * alpha > E.
//
// Backward phase, deepest level first: for every u at level L,
//   delta[u] = sigma[u] * sum over out-neighbours w at level L+1 of
//              (1 + delta[w]) / sigma[w]
// over the out-rows of level L's vertices, read where a bit says that the
// neighbour lies on level L+1 or deeper (out-neighbours of a level-L vertex lie
// at levels <= L+1), in the order of the level's list; the reached vertices
// are first put in (level, no out-edges, vertex ID) order, so the summation
// order is fixed and the results deterministic.  bc[u] += delta[u] for u !=
// source.
//
// What bounded the earlier form: on a 65 M-edge graph 43 ms for 12 sources, of
// them 24.5 on the GPU; the rest were 300 host reads of counts and 200 scratch
// allocations, each dear after such a read.  Now a level costs one host read
// (the next frontier's vertices, its out-edges and the vertices found, counted
// while they are found), none on the way back, and no allocation: the appends
// reserve a vertex's place in the list and its place among the frontier's
// out-edges with one 64-bit atomic, so the list comes with its prefix and
// needs no scan.  Edges find their row with a warp's row walk (rowwalk.cuh)
// instead of a binary search per edge in shared memory, the counts come through
// pinned words, and launches are chained.  12 sources: 43.4 -> 12.3 ms; 4 sources on
// 0.9 M edges: 7.6 -> 1.06 ms.
#include <algorithm>
#include <vector>

#include "carry_runs.cuh"
#include "handles.cuh"
#include "rowwalk.cuh"

struct cg_bc {
  int device = 0;
  int32_t V = 0;
  int64_t E = 0;
  const int64_t* in_off = nullptr;   // caller-owned in-edge CSR (pull)
  const int32_t* in_src = nullptr;
  const int64_t* out_off = nullptr;  // caller-owned out-edge CSR (push, backward)
  const int32_t* out_dst = nullptr;
  char* slab = nullptr;        // one allocation that holds the arrays below
  int32_t* level = nullptr;    // [V] BFS level of the current source (-1: unreached)
  double* sigma = nullptr;     // [V] shortest-path counts
  double* delta = nullptr;     // [V] dependencies
  double* xval = nullptr;      // [V] (1 + delta) / sigma, read where xbits says so
  double* acc = nullptr;       // [V] gathered sums, by list position
  uint32_t* xbits = nullptr;   // [V/32 + 1] one bit per vertex
  int32_t* flist[2] = {nullptr, nullptr};  // [V] a frontier's vertices that have out-edges
  int32_t* fpos[2] = {nullptr, nullptr};   // [V] their first places among its out-edges
  int32_t* fgap[2] = {nullptr, nullptr};   // [V] from those to their places in out_dst
  int32_t* lists = nullptr;    // [V] reached vertices, level after level
  int32_t* pos = nullptr;      // [V] row starts of `lists` (backward) or of `ids` (pull)
  int32_t* gap = nullptr;      // [V] from an edge's place among them to its place in the CSR
  int32_t* ids = nullptr;      // [V] unvisited vertices (pull); sort scratch
  uint32_t* keys = nullptr;    // [V] sort scratch
  uint32_t* keys_out = nullptr;  // [V]
  int64_t* tsum = nullptr;     // tile sums of a compaction and their prefix
  double* carry = nullptr;     // [E/256 + 2] open rows of the gather's tiles
  int32_t* carry_row = nullptr;
  unsigned long long* count = nullptr;  // [4] vertices << 32 | out-edges appended to the
                                        // frontier (three levels in turn), vertices reached
  void* sort = nullptr;        // scratch of the scans and the sort
  size_t sort_bytes = 0;
  unsigned long long* h_pin = nullptr;  // pinned host copy of count, and its ticket
  unsigned long long ticket = 0;
  double alpha = 16.0;
  int32_t depth = 0;           // levels of the last source
  int32_t last_source = -1;
  int32_t push_levels = 0, pull_levels = 0;
};

namespace cg {
namespace {

constexpr int kThreads = 256;
constexpr int kSub = 256;        // edges a warp folds at once: 8 consecutive per lane
constexpr int kPushTile = 256;   // frontier edges per warp in a push
typedef unsigned long long u64;

// Where a level's counts go when it is done: the host's pinned words, the
// ticket last.
struct Mailbox {
  u64* pin;
  u64 ticket;
};

__device__ __forceinline__ void publish(const u64* count, const Mailbox& box) {
  volatile u64* pin = box.pin;
  for (int q = 0; q < 4; ++q) pin[q] = __ldcg(count + q);
  __threadfence_system();
  pin[4] = box.ticket;
}

// The same by the last block of a launch (count[4]: blocks done, cleared
// again).  Every thread of the block calls it, when the block has counted.
__device__ __forceinline__ void publish_last(u64* count, const Mailbox& box) {
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(count + 4, 1ull) != gridDim.x - 1) return;
  __threadfence();
  count[4] = 0ull;
  publish(count, box);
}

__global__ void bc_reset_kernel(int32_t V, int32_t* level,
                                double* sigma, double* delta,
                                uint32_t* xbits) {
  if (!chain_begin()) return;
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    level[v] = -1;
    sigma[v] = 0.0;
    delta[v] = 0.0;
    if ((v & 31) == 0) xbits[v >> 5] = 0u;
  }
}

__device__ __forceinline__ void set_bit(uint32_t* bits, int32_t v, bool on) {
  if (on)
    atomicOr(bits + (v >> 5), 1u << (v & 31));
  else
    atomicAnd(bits + (v >> 5), ~(1u << (v & 31)));
}

__global__ void bc_seed_kernel(int32_t s, const int64_t* out_off,
                               int32_t* level, double* sigma,
                               int32_t* list, int32_t* fpos,
                               int32_t* fgap, u64* count, Mailbox box) {
  if (!chain_begin()) return;
  level[s] = 0;
  sigma[s] = 1.0;
  const u64 deg = (u64)(out_off[s + 1] - out_off[s]);
  list[0] = s;
  fpos[0] = 0;
  fgap[0] = (int32_t)out_off[s];
  count[0] = deg ? (1ull << 32) | deg : 0ull;
  count[1] = count[2] = count[4] = 0ull;
  count[3] = 1ull;
  __threadfence();
  publish(count, box);
}

struct Frontier {
  int32_t* list;
  int32_t* pos;
  int32_t* gap;
};

// The vertices found at this level by the warp: those with out-edges join the
// next frontier at places reserved together with their out-edges' places.
__device__ __forceinline__ void append(bool take, int32_t v, const int64_t* out_off,
                                       const Frontier& f, u64* next, u64* reached) {
  const unsigned full = 0xffffffffu;
  const unsigned found = __ballot_sync(full, take);
  if (!found) return;
  const int lane = threadIdx.x & 31;
  int64_t o0 = 0;
  int32_t deg = 0;
  if (take) {
    o0 = __ldca(out_off + v);
    deg = (int32_t)(__ldca(out_off + v + 1) - o0);
  }
  const unsigned m = __ballot_sync(full, deg > 0);
  int32_t incl = deg;  // a warp's degrees sum to at most E < 2^31 (its vertices are distinct)
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int32_t y = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += y;
  }
  u64 base = 0;
  if (lane == 31) {
    atomicAdd(reached, (u64)__popc(found));
    if (m) base = atomicAdd(next, ((u64)__popc(m) << 32) | (u64)(uint32_t)incl);
  }
  base = __shfl_sync(full, base, 31);
  if (deg > 0) {
    const int64_t at = (int64_t)(base >> 32) + __popc(m & ((1u << lane) - 1u));
    const int32_t p = (int32_t)(base & 0xffffffffull) + incl - deg;
    f.list[at] = v;
    f.pos[at] = p;
    f.gap[at] = (int32_t)o0 - p;
  }
}

// The same for a whole block (every thread calls it): one pair of atomics for
// its 256 vertices, where a warp's would queue up behind each other on the two
// counters.
__device__ __forceinline__ void append_block(bool take, int32_t v,
                                             const int64_t* out_off,
                                             const Frontier& f, u64* next, u64* reached) {
  __shared__ u64 s_w[kThreads / 32], s_base;
  __shared__ int s_found;
  const unsigned full = 0xffffffffu;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (!__syncthreads_or(take)) return;
  if (threadIdx.x == 0) s_found = 0;
  int64_t o0 = 0;
  u64 val = 0;
  if (take) {
    o0 = __ldca(out_off + v);
    const u64 deg = (u64)(__ldca(out_off + v + 1) - o0);
    if (deg) val = (1ull << 32) | deg;
  }
  u64 incl = val;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const u64 y = __shfl_up_sync(full, incl, o);
    if (lane >= o) incl += y;
  }
  if (lane == 31) s_w[w] = incl;
  const int found = __popc(__ballot_sync(full, take));
  __syncthreads();
  if (lane == 0 && found) atomicAdd(&s_found, found);
  __syncthreads();
  if (threadIdx.x == 0) {
    u64 total = 0;
    for (int q = 0; q < kThreads / 32; ++q) total += s_w[q];
    atomicAdd(reached, (u64)s_found);
    s_base = total ? atomicAdd(next, total) : 0ull;
  }
  __syncthreads();
  if (val) {
    u64 at = s_base + incl - val;
    for (int q = 0; q < w; ++q) at += s_w[q];
    const int32_t p = (int32_t)(at & 0xffffffffull);
    f.list[at >> 32] = v;
    f.pos[at >> 32] = p;
    f.gap[at >> 32] = (int32_t)o0 - p;
  }
  __syncthreads();  // s_w and s_base are used again
}

// Push: the frontier's n vertices and m out-edges, kPushTile edges per warp.
// The counts of the level after next are cleared for it.
__global__ void __launch_bounds__(kThreads)
push_kernel(Frontier cur, int32_t n, int32_t m, const int64_t* out_off,
            const int32_t* out_dst, int32_t L, int32_t* level,
            double* sigma, Frontier nxt, u64* count, Mailbox box) {
  if (!chain_begin()) return;
  u64* next = count + (L + 1) % 3;
  if (blockIdx.x == 0 && threadIdx.x == 0) count[(L + 2) % 3] = 0ull;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  DenseWalk walk(cur.pos, n, m);
  for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kPushTile; b < m;
       b += nw * kPushTile) {
    walk.seek((int32_t)b);
    for (int i = 0; i < kPushTile && b + i < m; i += 32) {
      const int64_t e = b + i + lane;
      int32_t j;
      walk.batch((int32_t)(b + i), &j);
      bool take = false;
      int32_t w = 0;
      if (e < m) {
        const int32_t u = __ldca(cur.list + j);
        w = __ldcs(out_dst + (e + __ldca(cur.gap + j)));
        // a target seen visited on an earlier level needs no atomic; one that
        // reads unvisited takes the compare-and-swap (it may lose to another
        // edge of this level, which then reads L + 1)
        int32_t old = __ldcg(level + w);
        if (old == -1) old = atomicCAS(level + w, -1, L + 1);
        take = old == -1;
        if (old == -1 || old == L + 1) atomicAdd(sigma + w, sigma[u]);
      }
      append(take, w, out_off, nxt, next, count + 3);
    }
  }
  publish_last(count, box);
}

// ---------------------------------------------------------------------------
// Compactions: a value per item, its exclusive prefix, and what to write there
// (tile sums, their scan, a second pass over the items).  What an item's writing
// needs (more) is read for all of a thread's items before any is written.
// ---------------------------------------------------------------------------
constexpr int kItems = 8;                      // per thread, 32 at a time per warp
constexpr int kCTile = kThreads * kItems;

// unvisited vertices that have in-edges: 1 << 32 | in-edges
struct Unvisited {
  const int32_t* level;
  const int64_t* in_off;
  int32_t* ids;
  int32_t* pos;
  int32_t* gap;
  __device__ u64 operator()(int64_t v) const {
    if (__ldca(level + v) != -1) return 0ull;
    const u64 d = (u64)(__ldca(in_off + v + 1) - __ldca(in_off + v));
    return d ? (1ull << 32) | d : 0ull;
  }
  __device__ int64_t more(int64_t v) const { return __ldca(in_off + v); }
  __device__ void put(int64_t v, int64_t row, u64 before) const {
    ids[before >> 32] = (int32_t)v;
    pos[before >> 32] = (int32_t)(before & 0xffffffffull);
    gap[before >> 32] = (int32_t)(row - (int64_t)(before & 0xffffffffull));
  }
};

// reached vertices, keyed by level and by having no out-edges
struct Reached {
  const int32_t* level;
  const int64_t* out_off;
  int32_t* ids;
  uint32_t* keys;
  __device__ u64 operator()(int64_t v) const { return __ldca(level + v) >= 0; }
  __device__ int64_t more(int64_t v) const {
    return (int64_t)__ldca(level + v) << 1 | (__ldca(out_off + v + 1) == __ldca(out_off + v));
  }
  __device__ void put(int64_t v, int64_t key, u64 before) const {
    ids[before] = (int32_t)v;
    keys[before] = (uint32_t)key;
  }
};

// row starts of the reached vertices in list order
struct ListRows {
  const int32_t* list;
  const int64_t* out_off;
  int32_t* pos;
  int32_t* gap;
  __device__ u64 operator()(int64_t i) const {
    const int32_t u = __ldca(list + i);
    return (u64)(__ldca(out_off + u + 1) - __ldca(out_off + u)) | 1ull << 63;
  }
  __device__ int64_t more(int64_t i) const { return __ldca(out_off + __ldca(list + i)); }
  __device__ void put(int64_t i, int64_t row, u64 before) const {
    const int32_t p = (int32_t)(before & 0x7fffffffull);
    pos[i] = p;
    gap[i] = (int32_t)row - p;
  }
};

template <class F, bool WRITE>
__global__ void __launch_bounds__(kThreads)
compact_kernel(F f, int64_t n, int64_t* tsum) {
  if (!chain_begin()) return;
  __shared__ u64 s_w[kThreads / 32];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kCTile + (int64_t)w * (kItems * 32);
  u64 v[kItems], sum = 0;
  int64_t more[WRITE ? kItems : 1];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int64_t i = base + r * 32 + lane;
    v[r] = i < n ? f(i) : 0ull;
    if (WRITE) more[r] = v[r] ? f.more(i) : 0;
    sum += v[r] & ~(1ull << 63);
  }
  for (int o = 16; o; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  if (lane == 0) s_w[w] = sum;
  __syncthreads();
  if (!WRITE) {
    if (threadIdx.x == 0) {
      u64 t = 0;
      for (int q = 0; q < kThreads / 32; ++q) t += s_w[q];
      tsum[blockIdx.x] = (int64_t)t;
    }
    return;
  }
  u64 run = (u64)tsum[blockIdx.x];
  for (int q = 0; q < w; ++q) run += s_w[q];
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const u64 x = v[r] & ~(1ull << 63);
    u64 incl = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const u64 y = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += y;
    }
    if (v[r]) f.put(base + r * 32 + lane, more[r], run + incl - x);
    run += __shfl_sync(0xffffffffu, incl, 31);
  }
}

// *total (device) = the values' sum.
template <class F>
int compact(cg_bc* h, const F& f, int64_t n, const int64_t** total, cudaStream_t s) {
  const int64_t tiles = ceil_div(n, kCTile);
  int64_t* scan = h->tsum + tiles;
  CG_TRY(launch_chained(compact_kernel<F, false>, (unsigned)tiles, kThreads, 0, s, f, n, h->tsum));
  Scratch ws(s, h->sort, h->sort_bytes);
  CG_TRY(exclusive_scan_i64(h->tsum, scan, tiles, s, &ws));
  CG_TRY(launch_chained(compact_kernel<F, true>, (unsigned)tiles, kThreads, 0, s, f, n, scan));
  if (total) *total = scan + tiles;
  return CG_OK;
}

// ---------------------------------------------------------------------------
// Row sums: out[i] = sum over the edges of listed row i (every listed row has an
// edge; its neighbours lie in vadj, gap[i] behind their places among the
// listed rows' edges laid end to end) of x at the neighbours whose bit is set.  A warp takes a tile of 256 or 1024 consecutive
// edges (pos: the rows' starts among them): it looks 32 edges at a time up, keeps the 256 values in shared memory, and then folds 8 consecutive ones
// per lane, one segmented scan joining the lanes.  FP64 adds run at 2 per
// cycle and SM here, so there are 13 warp adds per 256 edges and no more; the
// loads behind them are the adjacency stream and, per edge, a bit (V / 8
// bytes: stays on chip).  The largest levels of a 65 M-edge graph: 577 -> 300 us
// (a search per edge by shuffles took 1000 instructions per 256 edges and 490
// us; the list's rows all have edges, so a bit mask of their ends does).  A row that is open at a tile's end leaves its part
// in the tile's carry (completed in order by row_fix_kernel).
// ---------------------------------------------------------------------------
struct RowSums {
  const int32_t* pos;
  const int32_t* gap;
  int32_t origin;          // pos of row 0
  int64_t n, m;            // rows and edges, or
  const int64_t* packed;   // rows << 32 | edges on the device
  const int32_t* vadj;
  const uint32_t* bits;
  const double* x;
  double* out;
  double* carry;
  int32_t* carry_row;
  __device__ __forceinline__ int64_t rows() const { return packed ? *packed >> 32 : n; }
  __device__ __forceinline__ int64_t edges() const {
    return packed ? *packed & 0xffffffffll : m;
  }
};

// 256-edge steps of a tile: few long tiles where there is work for every warp
__device__ __forceinline__ int tile_steps(int64_t m) { return m >= ((int64_t)1 << 22) ? 4 : 1; }

__device__ __forceinline__ int pad8(int j) { return j + (j >> 3); }

// (All 8 batches' reads in flight, 5 blocks per SM: the 100 launches of 12 sources
// at 65 M edges 7.42 ms with 64-bit places, 4 batches and 4 blocks, 6.55 so; 6
// blocks and 4 batches 6.54, 6 and 8 spill, 6.79.)
__global__ void __launch_bounds__(kThreads, 5)
row_sum_kernel(RowSums a) {
  if (!chain_begin()) return;
  __shared__ double s_all[kThreads / 32][kSub + kSub / 8];
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int U = 8;  // batches of 32 edges whose reads are in flight together
  const int lane = threadIdx.x & 31;
  double* sv = s_all[threadIdx.x >> 5];
  // places among the listed rows' edges and in the CSR are below 2^31 - 1
  const uint32_t m = (uint32_t)a.edges();
  const uint32_t tile = (uint32_t)(tile_steps(m) * kSub), ntiles = (m + tile - 1) / tile;
  const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
  const int32_t* vadj = a.vadj + a.origin;
  DenseWalk walk(a.pos, (int32_t)a.rows(), (int32_t)m, a.origin);
  for (uint32_t t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < ntiles; t += nw) {
    const uint32_t t0 = t * tile, t1 = min(t0 + tile, m);
    walk.seek((int32_t)t0);
    double open = 0.0;       // the part so far of the row open before the step
    int32_t open_row = -1;   // the row open behind it
    for (uint32_t b = t0; b < t1; b += kSub) {
      uint32_t ends = 0;     // lane q < 8: the row ends of batch q
      int32_t row0 = 0;      // row of the step's first edge
#pragma unroll
      for (int q0 = 0; q0 < kSub / 32; q0 += U) {
        int32_t w[U];
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const uint32_t e = b + (q0 + u) * 32 + lane;
          int32_t r;
          if (q0 + u == 0) row0 = walk.row;
          const uint32_t f = walk.batch((int32_t)(b + (q0 + u) * 32), &r);
          if (lane == q0 + u) ends = f;
          w[u] = e < t1 ? (int32_t)e + __ldca(a.gap + r) : -1;  // place in vadj
        }
#pragma unroll
        for (int u = 0; u < U; ++u) {
          const bool ok = b + (q0 + u) * 32 + lane < t1;
          w[u] = ok ? __ldcs(vadj + w[u]) : -1;
        }
        bool hit[U];
#pragma unroll
        for (int u = 0; u < U; ++u)
          hit[u] = w[u] >= 0 && ((__ldca(a.bits + (w[u] >> 5)) >> (w[u] & 31)) & 1u);
#pragma unroll
        for (int u = 0; u < U; ++u)
          sv[pad8((q0 + u) * 32 + lane)] = hit[u] ? __ldca(a.x + w[u]) : 0.0;
      }
      __syncwarp();
      const uint32_t fl = (__shfl_sync(kFull, ends, lane >> 2) >> (8 * (lane & 3))) & 0xFFu;
      const int F = __popc(fl);
      int incl = F;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
      }
      const int32_t first = row0 + incl - F;  // rows follow one another: each has an edge
      double acc = lane == 0 ? open : 0.0, first_val = 0.0;
      int nf = 0;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double v = sv[pad8(lane * 8 + u)];
        if (__double_as_longlong(v) != 0) acc += v;  // (an FP64 compare takes the adds' pipe)
        if (fl & (1u << u)) {
          if (nf == 0)
            first_val = acc;
          else
            a.out[first + nf] = acc;
          ++nf;
          acc = 0.0;
        }
      }
      double S = acc;
      int g = F > 0;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const double y = __shfl_up_sync(kFull, S, o);
        const int gy = __shfl_up_sync(kFull, g, o);
        if (lane >= o) {
          if (!g && __double_as_longlong(y) != 0) S = y + S;
          g |= gy;
        }
      }
      const double P = __shfl_up_sync(kFull, S, 1);
      if (F > 0) a.out[first] = lane > 0 ? P + first_val : first_val;
      open = __shfl_sync(kFull, S, 31);
      // the step's last edge: does its row end there?
      const int last = (int)(min(b + kSub, t1) - b) - 1;
      const uint32_t lw = __shfl_sync(kFull, ends, last >> 5);
      open_row = (lw >> (last & 31)) & 1u ? -1 : row0 + __shfl_sync(kFull, incl, 31);
      __syncwarp();
    }
    if (lane == 0) {
      a.carry[t] = open;
      a.carry_row[t] = open_row;
    }
  }
}

__global__ void __launch_bounds__(256) row_fix_kernel(RowSums a) {
  if (!chain_begin()) return;
  const int64_t m = a.edges();
  const int64_t tile = (int64_t)tile_steps(m) * kSub;
  fix_runs<SumF64>(a.carry_row, a.carry, (m + tile - 1) / tile, a.out);
}

int row_sums(const RowSums& a, int64_t most_edges, cudaStream_t s) {
  const int64_t tiles = ceil_div(most_edges, kSub);
  CG_TRY(launch_chained(row_sum_kernel, grid_for(tiles * 32, kThreads, 5), kThreads, 0, s, a));
  if (tiles > 1)  // (one tile ends with its last row)
    CG_TRY(launch_chained(row_fix_kernel, grid_for(tiles, 256, 4), 256, 0, s, a));
  return CG_OK;
}

// After the pull's sums: one with a non-zero sum (a frontier in-neighbour) is on
// level L+1.
__global__ void __launch_bounds__(kThreads)
pull_update_kernel(const int32_t* ids, const int64_t* packed,
                   const double* acc, const int64_t* out_off, int32_t L,
                   int32_t* level, double* sigma, Frontier nxt,
                   u64* count, Mailbox box) {
  if (!chain_begin()) return;
  u64* next = count + (L + 1) % 3;
  if (blockIdx.x == 0 && threadIdx.x == 0) count[(L + 2) % 3] = 0ull;
  const int64_t n = *packed >> 32;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x; i0 < n; i0 += stride) {
    const int64_t i = i0 + threadIdx.x;  // the block stays together for the append
    bool take = false;
    int32_t v = 0;
    if (i < n) {
      v = ids[i];
      const double x = acc[i];
      if (x != 0.0) {
        level[v] = L + 1;
        sigma[v] = x;
        take = true;
      }
    }
    append_block(take, v, out_off, nxt, next, count + 3);
  }
  publish_last(count, box);
}

__global__ void set_bits_kernel(const int32_t* list, int64_t n,
                                uint32_t* bits, bool on) {
  if (!chain_begin()) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    set_bit(bits, list[i], on);
}

// A level's n listed vertices, the first `summed` of them with gathered sums (0
// for the others): delta, bc += delta (not for the source) and x = (1 + delta)
// / sigma for the next level up.
__global__ void dependency_kernel(const int32_t* list, int64_t n, int64_t summed,
                                  const double* sums, const double* sigma,
                                  double* delta, double* xval,
                                  uint32_t* xbits, double* bc,
                                  int32_t source) {
  if (!chain_begin()) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t u = list[i];
    const double sg = sigma[u];
    double d = 0.0;
    if (i < summed) {
      const double before = bc[u];
      d = sg * sums[i];
      delta[u] = d;
      if (u != source) bc[u] = before + d;
    }
    xval[u] = (1.0 + d) / sg;
    set_bit(xbits, u, true);
  }
}

__global__ void row_of_edge_kernel(const int64_t* __restrict__ off, int32_t V, int64_t E,
                                   int32_t* __restrict__ dst) {
  constexpr int kTile = 1024;
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  RowWalk<int64_t> walk(off, V, (int32_t)E);
  for (int64_t b = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * kTile; b < E;
       b += nw * kTile) {
    walk.seek((int32_t)b);
    for (int i = 0; i < kTile && b + i < E; i += 32) {
      const int64_t e = b + i + lane;
      int32_t st, en;
      const int32_t r = walk.row_of((int32_t)e, e < E, &st, &en);
      if (e < E) __stcs(dst + e, r);
    }
  }
}

// Waits for the counts of the last mailbox.
int wait_counts(cg_bc* h, cudaStream_t s) {
  return wait_ticket(h->h_pin + 4, h->ticket, s, "bc_run");
}

// The mailbox of the launch that is next to be waited for.
Mailbox mailbox(cg_bc* h) { return Mailbox{h->h_pin, ++h->ticket}; }

Frontier frontier(const cg_bc* h, int q) { return Frontier{h->flist[q], h->fpos[q], h->fgap[q]}; }

// One bottom-up level: the unvisited vertices that have in-edges, in ID order,
// gather sigma of the frontier's n vertices over their in-rows.  Visited
// vertices' rows are never read.
int pull_level(cg_bc* h, int32_t L, int32_t n, cudaStream_t s) {
  const int32_t V = h->V;
  const int cur = L & 1;
  CG_TRY(launch_chained(set_bits_kernel, grid_for(n, kThreads), kThreads, 0, s, h->flist[cur], n,
                        h->xbits, true));
  const int64_t* packed = nullptr;
  CG_TRY(compact(h, Unvisited{h->level, h->in_off, h->ids, h->pos, h->gap}, V, &packed, s));
  const RowSums a{h->pos, h->gap, 0, 0, 0, packed, h->in_src, h->xbits, h->sigma, h->acc,
                  h->carry, h->carry_row};
  CG_TRY(row_sums(a, h->E, s));
  CG_TRY(launch_chained(pull_update_kernel, grid_for(V, kThreads), kThreads, 0, s, h->ids, packed,
                        h->acc, h->out_off, L, h->level, h->sigma, frontier(h, 1 - cur),
                        h->count, mailbox(h)));
  CG_TRY(launch_chained(set_bits_kernel, grid_for(n, kThreads), kThreads, 0, s, h->flist[cur], n,
                        h->xbits, false));
  return CG_OK;
}

int run_source(cg_bc* h, int32_t src, double* bc, cudaStream_t s) {
  const int32_t V = h->V;
  CG_TRY(launch_chained(bc_reset_kernel, grid_for(V, kThreads), kThreads, 0, s, V, h->level,
                        h->sigma, h->delta, h->xbits));
  CG_TRY(launch_chained(bc_seed_kernel, 1, 1, 0, s, src, h->out_off, h->level, h->sigma,
                        h->flist[0], h->fpos[0], h->fgap[0], h->count, mailbox(h)));
  CG_TRY(wait_counts(h, s));
  // per level: vertices, of them with out-edges, and these edges
  std::vector<int64_t> size(1, 1), rows, edges;
  h->push_levels = h->pull_levels = 0;
  // forward: one level per round until a level adds nobody
  for (int32_t L = 0;; ++L) {
    const u64 packed = h->h_pin[L % 3], reached = h->h_pin[3];
    const int32_t n = (int32_t)(packed >> 32), m = (int32_t)(packed & 0xffffffffull);
    rows.push_back(n);
    edges.push_back(m);
    if (m == 0) break;  // L is the deepest level
    if ((double)m * h->alpha > (double)h->E) {  // pull (bottom-up)
      CG_TRY(pull_level(h, L, n, s));
      ++h->pull_levels;
    } else {  // push from the frontier's out-edges
      const int cur = L & 1;
      CG_TRY(launch_chained(push_kernel, grid_for(ceil_div(m, kPushTile) * 32, kThreads), kThreads,
                            0, s, frontier(h, cur), n, m, h->out_off, h->out_dst, L, h->level,
                            h->sigma, frontier(h, 1 - cur), h->count, mailbox(h)));
      ++h->push_levels;
    }
    CG_TRY(wait_counts(h, s));
    if (h->h_pin[3] == reached) break;  // nothing new
    size.push_back((int64_t)(h->h_pin[3] - reached));
  }
  const int32_t depth = (int32_t)size.size();  // levels 0 .. depth-1
  h->depth = depth;
  int64_t reached = 0;
  for (int64_t q : size) reached += q;
  // the reached vertices in (level, no out-edges, ID) order, and their row starts
  CG_TRY(compact(h, Reached{h->level, h->out_off, h->ids, h->keys}, V, nullptr, s));
  int bits = 1;
  while (bits < 32 && (int64_t(1) << bits) < 2 * (int64_t)depth) ++bits;
  {
    Scratch ws(s, h->sort, h->sort_bytes);
    CG_TRY(radix_sort_pairs(h->keys, h->ids, h->keys_out, h->lists, reached, bits, s, &ws));
  }
  CG_TRY(compact(h, ListRows{h->lists, h->out_off, h->pos, h->gap}, reached, nullptr, s));
  // backward: the deepest level, whose sums are all 0, then levels depth-2 .. 0
  int64_t b0 = reached, e0 = 0;
  for (int32_t L = 0; L < depth; ++L) e0 += edges[L];
  for (int32_t L = depth - 1; L >= 0; --L) {
    const int64_t n = size[L];
    b0 -= n;
    e0 -= edges[L];
    const int32_t* list = h->lists + b0;
    int64_t summed = 0;
    if (L < depth - 1) {
      summed = rows[L];
      const RowSums a{h->pos + b0, h->gap + b0, (int32_t)e0, rows[L], edges[L], nullptr,
                      h->out_dst, h->xbits, h->xval, h->acc, h->carry, h->carry_row};
      CG_TRY(row_sums(a, edges[L], s));
    }
    CG_TRY(launch_chained(dependency_kernel, grid_for(n, kThreads), kThreads, 0, s, list, n,
                          summed, h->acc, h->sigma, h->delta, h->xval, h->xbits, bc, src));
  }
  h->last_source = src;
  return CG_OK;
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int cg_transpose_csr(const int64_t* in_offsets, const int32_t* in_src, int32_t V, int64_t E,
                     int64_t* out_offsets, int32_t* out_dst, cudaStream_t stream) {
  CG_ARG(V >= 1 && E >= 0 && E < 0x7FFFFFFFLL, "cg_transpose_csr: V >= 1 and 0 <= E < 2^31-1");
  CG_ARG(in_offsets && out_offsets && (E == 0 || (in_src && out_dst)),
         "cg_transpose_csr: null pointer argument");
  CG_TRY(validate_csr(in_offsets, in_src, V, E, stream));
  int32_t* deg = nullptr;
  int32_t* rows = nullptr;
  uint32_t* kout = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&deg, sizeof(int32_t) * (size_t)V, stream);
  int st = e == cudaSuccess ? CG_OK : cuda_fail(e, "cg_transpose_csr", __FILE__, __LINE__);
  if (st == CG_OK) st = cg_out_degree(in_src, E, V, deg, stream);
  if (st == CG_OK) st = exclusive_scan_i32_to_i64(deg, out_offsets, V, stream);
  if (st == CG_OK && E > 0) {
    e = cudaMallocAsync((void**)&rows, sizeof(int32_t) * (size_t)E, stream);
    if (e == cudaSuccess) e = cudaMallocAsync((void**)&kout, sizeof(uint32_t) * (size_t)E, stream);
    if (e == cudaSuccess) {
      row_of_edge_kernel<<<grid_for(ceil_div(E, 1024) * 32, 256), 256, 0, stream>>>(in_offsets, V,
                                                                                    E, rows);
      e = cudaGetLastError();
    }
    if (e != cudaSuccess) st = cuda_fail(e, "cg_transpose_csr", __FILE__, __LINE__);
    int bits = 1;
    while (bits < 32 && (int64_t(1) << bits) < (int64_t)V) ++bits;
    // stable sort of the edges by source keeps each out-row in ascending
    // destination order (the in-edge CSR lists its rows in that order)
    if (st == CG_OK)
      st = radix_sort_pairs(reinterpret_cast<const uint32_t*>(in_src), rows, kout, out_dst, E,
                            bits, stream);
  }
  if (deg) cudaFreeAsync(deg, stream);
  if (rows) cudaFreeAsync(rows, stream);
  if (kout) cudaFreeAsync(kout, stream);
  return st;
}

int bc_create(const int64_t* in_offsets, const int32_t* in_src, const int64_t* out_offsets,
              const int32_t* out_dst, int32_t V, int64_t E, cg_bc** out, cudaStream_t stream) {
  CG_ARG(out != nullptr, "bc_create: out is NULL");
  *out = nullptr;
  CG_ARG(V >= 1 && E >= 0 && E < 0x7FFFFFFFLL, "bc_create: V >= 1 and 0 <= E < 2^31-1");
  CG_ARG(in_offsets && out_offsets && (E == 0 || (in_src && out_dst)),
         "bc_create: null pointer argument");
  CG_TRY(validate_csr(in_offsets, in_src, V, E, stream));
  CG_TRY(validate_csr(out_offsets, out_dst, V, E, stream));
  cg_bc* h = new cg_bc();
  cudaGetDevice(&h->device);
  h->V = V;
  h->E = E;
  h->in_off = in_offsets;
  h->in_src = in_src;
  h->out_off = out_offsets;
  h->out_dst = out_dst;
  const size_t v4 = Scratch::round(4 * (size_t)V), v8 = Scratch::round(8 * (size_t)V);
  const int64_t tiles = ceil_div(V, kCTile);
  const size_t nc = (size_t)(E / kSub + 2);
  h->sort_bytes = sort_scratch(V) + scan_scratch(tiles) + 4096;
  const size_t ts = Scratch::round(8 * (size_t)(2 * tiles + 2));
  const size_t xb = Scratch::round(4 * ((size_t)V / 32 + 1));
  const size_t c8 = Scratch::round(8 * nc), c4 = Scratch::round(4 * nc);
  cudaError_t e = cudaMalloc((void**)&h->slab, 13 * v4 + 4 * v8 + xb + ts + c8 + c4 + 256 +
                                                   h->sort_bytes);
  if (e == cudaSuccess) {
    char* p = h->slab;
    auto take = [&](size_t bytes) {
      char* q = p;
      p += bytes;
      return q;
    };
    h->sigma = reinterpret_cast<double*>(take(v8));
    h->delta = reinterpret_cast<double*>(take(v8));
    h->xval = reinterpret_cast<double*>(take(v8));
    h->acc = reinterpret_cast<double*>(take(v8));
    h->level = reinterpret_cast<int32_t*>(take(v4));
    for (int q = 0; q < 2; ++q) {
      h->flist[q] = reinterpret_cast<int32_t*>(take(v4));
      h->fpos[q] = reinterpret_cast<int32_t*>(take(v4));
      h->fgap[q] = reinterpret_cast<int32_t*>(take(v4));
    }
    h->lists = reinterpret_cast<int32_t*>(take(v4));
    h->pos = reinterpret_cast<int32_t*>(take(v4));
    h->gap = reinterpret_cast<int32_t*>(take(v4));
    h->ids = reinterpret_cast<int32_t*>(take(v4));
    h->keys = reinterpret_cast<uint32_t*>(take(v4));
    h->keys_out = reinterpret_cast<uint32_t*>(take(v4));
    h->xbits = reinterpret_cast<uint32_t*>(take(xb));
    h->tsum = reinterpret_cast<int64_t*>(take(ts));
    h->carry = reinterpret_cast<double*>(take(c8));
    h->carry_row = reinterpret_cast<int32_t*>(take(c4));
    h->count = reinterpret_cast<unsigned long long*>(take(256));
    h->sort = take(h->sort_bytes);
    e = cudaHostAlloc((void**)&h->h_pin, 5 * sizeof(unsigned long long), 0);
    if (e == cudaSuccess) std::fill(h->h_pin, h->h_pin + 5, 0ull);
  }
  int st = e == cudaSuccess ? CG_OK : cuda_fail(e, "bc_create", __FILE__, __LINE__);
  if (st == CG_OK) {
    e = cudaStreamSynchronize(stream);
    if (e != cudaSuccess) st = cuda_fail(e, "bc_create", __FILE__, __LINE__);
  }
  if (st != CG_OK) {
    bc_destroy(h);
    return st;
  }
  *out = h;
  return CG_OK;
}

int bc_destroy(cg_bc* h) {
  if (!h) return CG_OK;
  int cur = 0;
  cudaGetDevice(&cur);
  if (cur != h->device) cudaSetDevice(h->device);
  cudaDeviceSynchronize();
  cudaFree(h->slab);
  if (h->h_pin) cudaFreeHost(h->h_pin);
  if (cur != h->device) cudaSetDevice(cur);
  delete h;
  return CG_OK;
}

int bc_set_direction(cg_bc* h, double alpha) {
  CG_ARG(h != nullptr, "bc_set_direction: null handle");
  CG_ARG(alpha >= 0.0, "bc_set_direction: alpha must be >= 0");
  h->alpha = alpha;
  return CG_OK;
}

int bc_run(cg_bc* h, const int32_t* sources, int32_t nsources, double* bc, cudaStream_t stream) {
  CG_ARG(h != nullptr, "bc_run: null handle");
  CG_ARG(nsources >= 0 && (nsources == 0 || sources) && bc, "bc_run: bad arguments");
  for (int32_t i = 0; i < nsources; ++i)
    CG_ARG(sources[i] >= 0 && sources[i] < h->V, "bc_run: source %d outside [0, %d)",
           sources[i], h->V);
  for (int32_t i = 0; i < nsources; ++i) CG_TRY(run_source(h, sources[i], bc, stream));
  return CG_OK;
}

int bc_source_state(const cg_bc* h, int32_t* level, double* sigma, double* delta,
                    int32_t* depth, int32_t* push_levels, int32_t* pull_levels,
                    cudaStream_t stream) {
  CG_ARG(h != nullptr, "bc_source_state: null handle");
  CG_ARG(h->last_source >= 0, "bc_source_state: no source has run yet");
  const size_t v4 = sizeof(int32_t) * (size_t)h->V, v8 = sizeof(double) * (size_t)h->V;
  if (level) CG_CUDA(cudaMemcpyAsync(level, h->level, v4, cudaMemcpyDeviceToDevice, stream));
  if (sigma) CG_CUDA(cudaMemcpyAsync(sigma, h->sigma, v8, cudaMemcpyDeviceToDevice, stream));
  if (delta) CG_CUDA(cudaMemcpyAsync(delta, h->delta, v8, cudaMemcpyDeviceToDevice, stream));
  if (depth) *depth = h->depth;
  if (push_levels) *push_levels = h->push_levels;
  if (pull_levels) *pull_levels = h->pull_levels;
  return CG_OK;
}

}  // extern "C"
