// CSR segmenting preprocessing (Algorithm 2, Section III-A) on the GPU.
//
// 65.2 M edges in 7 segments: 1.1 ms of kernels, against 8.4 ms for the
// warp-per-row passes this replaces (which counted, listed and sorted (row,
// segment) pairs with most lanes idle on short rows).
//
// Steps (all device work except reading a few sizes back).  Algorithm 2 is a
// stable split of the edges, which lie in (destination, parent) order, by
// their source's segment:
//   A. per tile of edges, how many go to each segment; a scan over (segment,
//      tile) gives every tile its places, and the segments' edge ranges;
//   B. the tiles' sources and destinations move to those places;
//   C. a subgraph row begins where the destination or the segment changes: a
//      count and a scan number the rows, and one pass writes idxMap, the row
//      starts and the flagged segment-local sources;
//   D. merge-block indices (blockStarts / blockEnds of Algorithm 4);
//   E. the gather tiling and the intermBuf of the handle.
#include <algorithm>
#include <numeric>
#include <vector>

#include "handles.cuh"
#include "rowwalk.cuh"

namespace cg {
namespace {

constexpr int kMaxSegments = 1024;
constexpr int32_t kFewDegrees = 1 << 16;  // see pr_plan_bounds
constexpr int kSplitThreads = 256;
constexpr int kSplitWarps = kSplitThreads / 32;
constexpr int kSplitRounds = 8;                               // edges per thread
constexpr int kSplitTile = kSplitThreads * kSplitRounds;      // 2048
constexpr int kSplitBlocks = 4;  // blocks per SM: 64 registers per thread
constexpr uint32_t kSegmentStart = 0x80000000u;               // first edge of a segment

// Segment of source u: last s with bounds[s] <= u (empty segments skipped).
__device__ __forceinline__ int seg_of(int32_t u, const int32_t* sb, int k) {
  int lo = 0, hi = k + 1;  // upper_bound over sb[0..k]
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (sb[mid] <= u) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

__global__ void validate_csr_kernel(const int64_t* __restrict__ offsets,
                                    const int32_t* __restrict__ src, int32_t V, int64_t E,
                                    unsigned long long* __restrict__ bad) {
  unsigned long long nbad = 0;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t t0 = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  for (int64_t v = t0; v < V; v += stride) nbad += offsets[v + 1] < offsets[v];
  if (t0 == 0) nbad += (offsets[0] != 0) + (offsets[V] != E);
  for (int64_t e = t0; e < E; e += stride) {
    const int32_t u = __ldcs(src + e);
    nbad += (u < 0 || u >= V);
  }
  nbad = warp_sum(nbad);
  if ((threadIdx.x & 31) == 0 && nbad) atomicAdd(bad, nbad);
}

// A + B.  A warp owns 256 consecutive edges of the tile, visited 32 at a time,
// so (warp, round, lane) order is the edges' order; equal segments of a round
// are ranked with __match_any_sync.  Without SCATTER only the tile's counts
// are written (counts[s * ntiles + tile]).
template <bool SCATTER>
__global__ void __launch_bounds__(kSplitThreads, kSplitBlocks)
split_kernel(const int64_t* __restrict__ offsets, const int32_t* __restrict__ src, int32_t V,
             int64_t E, const int32_t* __restrict__ bounds, int k, int64_t ntiles,
             int32_t* __restrict__ counts, const int64_t* __restrict__ place,
             const int64_t* __restrict__ edge_base, const int64_t* __restrict__ cstart,
             uint32_t* __restrict__ colf, uint32_t* __restrict__ sdst) {
  extern __shared__ int32_t sm[];
  int32_t* sb = sm;             // [k+1]
  int32_t* wc = sb + (k + 1);   // [warps][k]
  int32_t* pl = wc + kSplitWarps * k;  // [k] the tile's first place in each segment
  int32_t* gap = pl + k;               // [k] from an edge's place to its place in colf
  for (int i = threadIdx.x; i <= k; i += kSplitThreads) sb[i] = bounds[i];
  for (int i = threadIdx.x; i < kSplitWarps * k; i += kSplitThreads) wc[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const unsigned lt = (1u << lane) - 1u;
  const int64_t base = (int64_t)blockIdx.x * kSplitTile + (int64_t)w * (kSplitRounds * 32);
  int32_t* mine = wc + w * k;
  int32_t u[kSplitRounds];
  int32_t sr[SCATTER ? kSplitRounds : 1];  // segment << 16 | rank in the warp
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const int64_t e = base + r * 32 + lane;
    u[r] = e < E ? __ldcs(src + e) : -1;
  }
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const bool ok = u[r] >= 0;
    const int s = ok ? seg_of(u[r], sb, k) : 0;
    const unsigned peers = __match_any_sync(0xffffffffu, ok ? (unsigned)s : 0x10000u);
    const int before = ok ? mine[s] : 0;
    if (SCATTER) sr[r] = (s << 16) | (before + __popc(peers & lt));
    __syncwarp();
    if (ok && lane == __ffs(peers) - 1) mine[s] = before + __popc(peers);
    __syncwarp();
  }
  __syncthreads();
  for (int s = threadIdx.x; s < k; s += kSplitThreads) {
    int32_t run = 0;
    for (int q = 0; q < kSplitWarps; ++q) {
      const int32_t t = wc[q * k + s];
      wc[q * k + s] = run;
      run += t;
    }
    if (!SCATTER)
      counts[(int64_t)s * ntiles + blockIdx.x] = run;
    else
    {
      pl[s] = (int32_t)place[(int64_t)s * ntiles + blockIdx.x];  // < E < 2^31
      gap[s] = (int32_t)(cstart[s] - edge_base[s]);
    }
  }
  if (!SCATTER) return;
  __syncthreads();
  if (base >= E) return;
  RowWalk<int64_t> walk(offsets, V, (int32_t)E);
  walk.seek((int32_t)base);
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const int64_t e = base + r * 32 + lane;
    int32_t st, en;
    const int32_t row = walk.row_of((int32_t)e, e < E, &st, &en);
    if (e < E) {
      const int s = sr[r] >> 16;
      const int32_t pos = pl[s] + mine[s] + (sr[r] & 0xFFFF);
      colf[pos + gap[s]] = (uint32_t)u[r];
      sdst[pos] = (uint32_t)row;
    }
  }
}

// The segments' edge ranges; their first edges, marked in sdst.
__global__ void split_base_kernel(const int64_t* __restrict__ place, int64_t ntiles, int k,
                                  int64_t E, int64_t* __restrict__ edge_base) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s <= k; s += gridDim.x * blockDim.x)
    edge_base[s] = s < k ? place[(int64_t)s * ntiles] : E;
}
__global__ void split_mark_kernel(const int64_t* __restrict__ edge_base, int k, int64_t E,
                                  uint32_t* __restrict__ sdst) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < k; s += gridDim.x * blockDim.x)
    if (edge_base[s] < E) atomicOr(sdst + edge_base[s], kSegmentStart);
}

// C.  Does a subgraph row begin at edge e (d: its destination word, p: the one
// before it)?
__device__ __forceinline__ bool row_begins(uint32_t d, uint32_t p) {
  return (d & kSegmentStart) || d != (p & ~kSegmentStart);
}

// Tiles of 2048 edges, a warp 256 consecutive ones.  Without WRITE: the tile's
// rows are counted.  With it (first: the tiles' exclusive prefix): idx_map and
// row starts, and every edge's global source in colf, in place, as
// segment-local source with its row-end flag.
template <bool WRITE>
__global__ void __launch_bounds__(kSplitThreads, kSplitBlocks)
rows_kernel(const uint32_t* __restrict__ sdst, int64_t E,
            int32_t* __restrict__ tile_rows, const int64_t* __restrict__ first,
            const int64_t* __restrict__ edge_base, const int64_t* __restrict__ cstart,
            const int64_t* __restrict__ bounds, int k, int32_t* __restrict__ idx_map,
            int32_t* __restrict__ row_ptr, uint32_t* colf) {
  __shared__ int32_t s_cnt[kSplitWarps];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t base = (int64_t)blockIdx.x * kSplitTile + (int64_t)w * (kSplitRounds * 32);
  uint32_t d[kSplitRounds], heads[kSplitRounds];
  uint32_t last = base > 0 && base < E ? __ldg(sdst + base - 1) : 0u;
  int cnt = 0;
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const int64_t e = base + r * 32 + lane;
    d[r] = e < E ? __ldcs(sdst + e) : 0u;
  }
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const uint32_t up = __shfl_up_sync(0xffffffffu, d[r], 1);
    const bool h = base + r * 32 + lane < E && row_begins(d[r], lane ? up : last);
    heads[r] = __ballot_sync(0xffffffffu, h);
    cnt += __popc(heads[r]);
    last = __shfl_sync(0xffffffffu, d[r], 31);
  }
  if (lane == 0) s_cnt[w] = cnt;
  __syncthreads();
  if (!WRITE) {
    if (threadIdx.x == 0) {
      int t = 0;
      for (int q = 0; q < kSplitWarps; ++q) t += s_cnt[q];
      tile_rows[blockIdx.x] = t;
    }
    return;
  }
  if (base >= E) return;
  int64_t row = first[blockIdx.x];
  for (int q = 0; q < w; ++q) row += s_cnt[q];
  // does a row begin right behind the warp's edges?
  const int64_t behind = base + kSplitRounds * 32;
  const bool next = behind >= E || row_begins(__ldg(sdst + behind), last);
  int s = -1;  // segment of the warp's first edge: the last s with edge_base[s] <= base
  for (int i = 0; i <= k; i += 32) {
    const bool le = i + lane <= k && __ldg(edge_base + i + lane) <= base;
    const unsigned m = __ballot_sync(0xffffffffu, le);
    s += __popc(m);
    if (m != 0xffffffffu) break;
  }
  int64_t send = __ldg(edge_base + s + 1);
  int64_t shift = __ldg(cstart + s) - __ldg(edge_base + s);
  int32_t src0 = (int32_t)__ldg(bounds + s);
  const bool plain = behind <= send;  // one segment, all edges there (behind <= send <= E)
  uint32_t c[kSplitRounds];
  if (plain) {
#pragma unroll
    for (int r = 0; r < kSplitRounds; ++r) c[r] = colf[base + r * 32 + lane + shift];
  }
#pragma unroll
  for (int r = 0; r < kSplitRounds; ++r) {
    const int64_t e = base + r * 32 + lane;
    const uint32_t h = heads[r];
    const uint32_t after = r + 1 < kSplitRounds ? heads[r + 1 < kSplitRounds ? r + 1 : r] & 1u
                                                : (uint32_t)next;
    if (e < E) {
      int64_t sh = shift;
      if (plain) {
        c[r] -= (uint32_t)src0;
      } else {  // a later segment may begin here
        int sl = s;
        while (e >= __ldg(edge_base + sl + 1)) ++sl;
        sh = __ldg(cstart + sl) - __ldg(edge_base + sl);
        c[r] = colf[e + sh] - (uint32_t)__ldg(bounds + sl);
      }
      if ((h >> lane) & 1u) {
        const int64_t i = row + __popc(h & ((1u << lane) - 1u));
        idx_map[i] = (int32_t)(d[r] & ~kSegmentStart);
        row_ptr[i] = (int32_t)e;
      }
      const bool ends = e == E - 1 || (lane < 31 ? (h >> (lane + 1)) & 1u : after);
      colf[e + sh] = c[r] | (ends ? kRowEndFlag : 0u);
    }
    row += __popc(h);
  }
}

// row_base[s] = first row at or behind the segment's first edge; the gaps
// behind the segments' edges in colf are cleared.
__global__ void segment_rows_kernel(const int32_t* __restrict__ row_ptr, int64_t rows, int k,
                                    const int64_t* __restrict__ edge_base,
                                    const int64_t* __restrict__ cstart, int64_t colf_len,
                                    int64_t* __restrict__ row_base, uint32_t* __restrict__ colf) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s <= k; s += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = rows;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (row_ptr[mid] < edge_base[s]) lo = mid + 1; else hi = mid;
    }
    row_base[s] = lo;
    const int64_t a = cstart[s] + (s < k ? edge_base[s + 1] - edge_base[s] : 0);
    const int64_t b = s < k ? cstart[s + 1] : colf_len;
    for (int64_t i = a; i < b; ++i) colf[i] = 0u;
  }
}

// D. merge-block indices, block-major: blk[b*k + s] = first row of segment s
// with destination >= b*B.
__global__ void blk_kernel(const int64_t* __restrict__ row_base, int k,
                           const int32_t* __restrict__ idx_map, int B, int nb,
                           int32_t* __restrict__ blk) {
  const int64_t n = (int64_t)k * (nb + 1);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t b = i / k, s = i - b * k;
    const int64_t v = b * B;
    int64_t lo = row_base[s], hi = row_base[s + 1];
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (idx_map[mid] < v) lo = mid + 1; else hi = mid;
    }
    blk[i] = (int32_t)lo;
  }
}

// sums[q] = out-edges of the vertices [q n, (q+1) n) for q < nr; sums[nr] = one
// past the last vertex with a non-zero degree.
__global__ void range_degree_kernel(const int32_t* __restrict__ deg, int32_t V, int32_t n,
                                    int64_t nr, int64_t* __restrict__ sums) {
  const int lane = threadIdx.x & 31;
  long long last = 0;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x; b < V; b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = b + threadIdx.x;
    const int32_t d = v < V ? __ldg(deg + v) : 0;
    if (d != 0) last = v + 1;
    const int64_t q = v / n, q0 = __shfl_sync(0xffffffffu, q, 0);
    if (__all_sync(0xffffffffu, q == q0)) {  // one range: one atomic per warp
      if (q0 >= nr) continue;
      const long long t = warp_sum((long long)d);
      if (lane == 0 && t != 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(sums + q0), (unsigned long long)t);
    } else if (d != 0 && q < nr) {
      atomicAdd(reinterpret_cast<unsigned long long*>(sums + q), (unsigned long long)(long long)d);
    }
  }
  for (int o = 16; o; o >>= 1) last = max(last, __shfl_xor_sync(0xffffffffu, last, o));
  if (lane == 0 && last)
    atomicMax(reinterpret_cast<unsigned long long*>(sums + nr), (unsigned long long)last);
}

// Export helpers.
__global__ void to_i64_kernel(const int32_t* __restrict__ in, int64_t n,
                              int64_t* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = in[i];
}

// Merge-block indices of the caller's block size, segment-major and local to
// the segment (out[s*(nb+1) + b]: rows of segment s with destination < b*B),
// the oracle's layout.
__global__ void blk_local_kernel(const int32_t* __restrict__ idx_map,
                                 const int64_t* __restrict__ rb, int k, int B, int nb,
                                 int32_t* __restrict__ out) {
  const int64_t n = (int64_t)k * (nb + 1);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t sg = i / (nb + 1), v = (i % (nb + 1)) * B;
    int64_t lo = rb[sg], hi = rb[sg + 1];
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (idx_map[mid] < v) lo = mid + 1; else hi = mid;
    }
    out[i] = (int32_t)(lo - rb[sg]);
  }
}

int build_impl(const int64_t* offsets, const int32_t* src, int32_t V, int64_t E, int32_t k,
               const std::vector<int64_t>& bounds, int32_t B, cg_segmented* g, cudaStream_t s) {
  const int64_t ntiles = ceil_div(E, kSplitTile);
  g->nb = (int32_t)ceil_div(V, B);
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  g->mB = merge_block(V, B, k, di.sm_count);
  g->mnb = (int32_t)ceil_div(V, g->mB);
  const size_t e4 = Scratch::round(4 * (size_t)E), kt = (size_t)k * ntiles;
  Scratch tmp(s, e4 + Scratch::round(4 * kt) + Scratch::round(8 * (kt + 1)) +
                     scan_scratch((int64_t)kt) + scan_scratch(ntiles) +
                     Scratch::round(8 * (size_t)(ntiles + 1)) + Scratch::round(4 * (size_t)ntiles) +
                     2 * Scratch::round(8 * (size_t)(k + 1)));
  int32_t *d_b32 = nullptr, *counts = nullptr, *tile_rows = nullptr;
  int64_t *place = nullptr, *d_eb = nullptr, *first = nullptr;
  uint32_t* sdst = nullptr;
  std::vector<int32_t> b32(bounds.begin(), bounds.end());
  g->edge_base.assign(k + 1, 0);
  g->row_base.assign(k + 1, 0);
  CG_CUDA(tmp.get(&d_b32, k + 1));
  CG_CUDA(tmp.get(&d_eb, k + 1));
  CG_CUDA(cudaMemcpyAsync(d_b32, b32.data(), sizeof(int32_t) * (k + 1), cudaMemcpyHostToDevice,
                          s));
  const size_t smem = sizeof(int32_t) * ((size_t)(k + 1) + (size_t)(kSplitWarps + 2) * k);
  if (E > 0) {  // A
    CG_CUDA(tmp.get(&counts, kt));
    CG_CUDA(tmp.get(&place, kt + 1));
    CG_CUDA(tmp.get(&sdst, E));
    CG_CUDA(tmp.get(&tile_rows, ntiles));
    CG_CUDA(tmp.get(&first, ntiles + 1));
    split_kernel<false><<<(unsigned)ntiles, kSplitThreads, smem, s>>>(
        offsets, src, V, E, d_b32, k, ntiles, counts, nullptr, nullptr, nullptr, nullptr, nullptr);
    CG_LAUNCH_CHECK();
    CG_TRY(exclusive_scan_i32_to_i64(counts, place, (int64_t)kt, s, &tmp));
    split_base_kernel<<<grid_for(k + 1, 128), 128, 0, s>>>(place, ntiles, k, E, d_eb);
    CG_LAUNCH_CHECK();
    CG_CUDA(cudaMemcpyAsync(g->edge_base.data(), d_eb, sizeof(int64_t) * (k + 1),
                            cudaMemcpyDeviceToHost, s));
  }
  CG_CUDA(cudaStreamSynchronize(s));  // edge_base
  CG_TRY(seg_plan_alloc(E, k, g->edge_base, bounds, &g->plan, s));
  if (g->plan.colf_len >= 0x7FFFFFFFLL) {  // the gathers keep places in it in 32 bits
    set_error("segmented gather: padded edge array exceeds 2^31 entries");
    return CG_ERR_UNSUPPORTED;
  }
  SegPlan* p = &g->plan;
  int64_t* d_rb = p->meta;
  int64_t* m_eb = p->meta + (k + 1);
  int64_t* m_cs = p->meta + 2 * (k + 1);
  int64_t* m_bd = p->meta + 3 * (k + 1);
  int64_t rows = 0;
  if (E > 0) {  // B, and C's count
    split_kernel<true><<<(unsigned)ntiles, kSplitThreads, smem, s>>>(
        offsets, src, V, E, d_b32, k, ntiles, nullptr, place, m_eb, m_cs, p->colf, sdst);
    CG_LAUNCH_CHECK();
    split_mark_kernel<<<grid_for(k, 128), 128, 0, s>>>(m_eb, k, E, sdst);
    CG_LAUNCH_CHECK();
    rows_kernel<false><<<(unsigned)ntiles, kSplitThreads, 0, s>>>(
        sdst, E, tile_rows, nullptr, nullptr, nullptr, nullptr, k, nullptr, nullptr, nullptr);
    CG_LAUNCH_CHECK();
    CG_TRY(exclusive_scan_i32_to_i64(tile_rows, first, ntiles, s, &tmp));
    CG_CUDA(cudaMemcpyAsync(&rows, first + ntiles, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
    CG_CUDA(cudaStreamSynchronize(s));
  }
  if (rows >= 0x7FFFFFFF) {
    set_error("pr_build_segments: %lld subgraph rows exceed the int32 range", (long long)rows);
    return CG_ERR_UNSUPPORTED;
  }
  g->rows = rows;
  // idx_map, row_ptr, blk and the iteration state (dslot, counter, partials,
  // rank_tmp, contrib_tmp, interm): one allocation
  const size_t n1 = (size_t)(rows > 0 ? rows : 1), nbk = (size_t)k * (g->mnb + 1);
  const size_t r4 = Scratch::round(4 * (n1 + 1));
  const size_t b4 = Scratch::round(4 * nbk), v4 = Scratch::round(4 * (size_t)V),
               pb = Scratch::round(16 * (size_t)g->mnb);
  CG_CUDA(cudaMalloc((void**)&g->idx_map, 2 * r4 + b4 + 256 + pb + 2 * v4 + 4 * n1));
  g->state = reinterpret_cast<char*>(g->idx_map) + 2 * r4 + b4;
  CG_CUDA(cudaMemsetAsync(g->state, 0, 256, s));
  g->row_ptr = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(g->idx_map) + r4);
  g->blk = reinterpret_cast<int32_t*>(reinterpret_cast<char*>(g->idx_map) + 2 * r4);
  const int32_t end = (int32_t)E;
  CG_CUDA(cudaMemcpyAsync(g->row_ptr + rows, &end, sizeof(int32_t), cudaMemcpyHostToDevice, s));
  if (E > 0) {
    rows_kernel<true><<<(unsigned)ntiles, kSplitThreads, 0, s>>>(
        sdst, E, nullptr, first, m_eb, m_cs, m_bd, k, g->idx_map, g->row_ptr, p->colf);
    CG_LAUNCH_CHECK();
  }
  segment_rows_kernel<<<grid_for(k + 1, 128), 128, 0, s>>>(g->row_ptr, rows, k, m_eb, m_cs,
                                                            p->colf_len, d_rb, p->colf);
  CG_LAUNCH_CHECK();
  CG_CUDA(cudaMemcpyAsync(g->row_base.data(), d_rb, sizeof(int64_t) * (k + 1),
                          cudaMemcpyDeviceToHost, s));
  // D
  blk_kernel<<<grid_for((int64_t)nbk, 256), 256, 0, s>>>(d_rb, k, g->idx_map, g->mB, g->mnb, g->blk);
  CG_LAUNCH_CHECK();
  CG_CUDA(cudaStreamSynchronize(s));  // row_base
  // E
  p->lent = sdst;  // done with: a second scratch of this size costs 0.6 ms at 65 M edges
  p->lent_bytes = E > 0 ? e4 : 0;
  const int st = seg_plan_finish(p, g->row_ptr, rows, g->row_base, s);
  p->lent = nullptr;
  p->lent_bytes = 0;
  CG_TRY(st);
  g->dslot = reinterpret_cast<double*>(g->state);
  g->counter = reinterpret_cast<unsigned*>(g->state + 128);
  g->partials = reinterpret_cast<double*>(g->state + 256);
  g->rank_tmp = reinterpret_cast<float*>(g->state + 256 + pb);
  g->contrib_tmp = reinterpret_cast<float*>(g->state + 256 + pb + v4);
  g->interm = g->state + 256 + pb + 2 * v4;
  g->bytes = 4 * (rows + 1) + 4 * rows + 4 * (int64_t)k * (g->mnb + 1) +
             seg_plan_bytes(g->plan) + 4 * rows + 16 * (int64_t)g->mnb + 4 + 32 + 8 * (int64_t)V;
  return CG_OK;
}

void free_segmented(cg_segmented* g) {
  if (g->pin) cudaFreeHost(g->pin);
  cudaFree(g->idx_map);
  seg_plan_free(&g->plan);
}

}  // namespace

int32_t merge_block(int32_t V, int32_t B, int32_t k, int sm_count) {
  const int64_t wave = (int64_t)sm_count * 40;
  auto in_waves = [&](int64_t w) {
    return std::min<int64_t>(B, ceil_div(ceil_div(V, w * wave), 32) * 32);
  };
  int64_t waves = ceil_div(ceil_div(V, B), wave);
  while (waves < 3 && in_waves(waves) * k > 3000) ++waves;
  return (int32_t)in_waves(waves);
}

int validate_csr(const int64_t* offsets, const int32_t* src, int32_t V, int64_t E,
                 cudaStream_t s) {
  Scratch tmp(s);
  unsigned long long* bad = nullptr;
  CG_CUDA(tmp.get(&bad, 1));
  cudaError_t e = cudaMemsetAsync(bad, 0, sizeof(unsigned long long), s);
  unsigned long long h = 0;
  if (e == cudaSuccess) {
    validate_csr_kernel<<<grid_for(std::max<int64_t>(V, E), 256), 256, 0, s>>>(offsets, src, V,
                                                                              E, bad);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(&h, bad, sizeof(h), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_fail(e, "validate_csr", __FILE__, __LINE__);
  if (h) {
    set_error("invalid CSR: %llu violations (offsets must rise from 0 to E; sources in [0, V))",
              h);
    return CG_ERR_INVALID_ARG;
  }
  return CG_OK;
}

}  // namespace cg

using namespace cg;

extern "C" {

int pr_build_segments(const int64_t* offsets, const int32_t* src, int32_t V, int64_t E,
                      int32_t k, const int64_t* host_bounds, int32_t B, cg_segmented** out,
                      cudaStream_t stream) {
  CG_ARG(out != nullptr, "pr_build_segments: out is NULL");
  *out = nullptr;
  CG_ARG(V >= 1, "pr_build_segments: V must be >= 1 (got %d)", V);
  CG_ARG(E >= 0 && E < 0x7FFFFFFFLL, "pr_build_segments: E must be in [0, 2^31-1)");
  CG_ARG(offsets && (E == 0 || src), "pr_build_segments: null CSR pointer");
  CG_ARG(k >= 1 && k <= kMaxSegments, "pr_build_segments: num_segments must be in [1, %d]",
         kMaxSegments);
  CG_ARG(B >= 1 && B <= 6144, "pr_build_segments: merge_block must be in [1, 6144]");
  std::vector<int64_t> bounds(k + 1);
  if (host_bounds) {
    for (int q = 0; q <= k; ++q) bounds[q] = host_bounds[q];
    CG_ARG(bounds[0] == 0 && bounds[k] == V, "pr_build_segments: bounds must run from 0 to V");
    for (int q = 0; q < k; ++q)
      CG_ARG(bounds[q] <= bounds[q + 1], "pr_build_segments: bounds must be non-decreasing");
  } else {
    const int64_t N = ceil_div(V, k);
    for (int q = 0; q <= k; ++q) bounds[q] = std::min<int64_t>((int64_t)q * N, V);
  }
  CG_TRY(validate_csr(offsets, src, V, E, stream));
  cg_segmented* g = new cg_segmented();
  CG_CUDA(cudaGetDevice(&g->device));
  g->V = V;
  g->E = E;
  g->k = k;
  g->B = B;
  g->bounds = bounds;
  int st = build_impl(offsets, src, V, E, k, bounds, B, g, stream);
  if (st != CG_OK) {
    cudaStreamSynchronize(stream);
    free_segmented(g);
    delete g;
    return st;
  }
  *out = g;
  return CG_OK;
}

int cg_segmented_get_info(const cg_segmented* g, cg_segmented_info* info) {
  CG_ARG(g && info, "cg_segmented_get_info: null pointer");
  info->V = g->V;
  info->E = g->E;
  info->num_segments = g->k;
  info->merge_block = g->B;
  info->num_blocks = g->nb;
  info->rows = g->rows;
  info->q = g->V ? (double)g->rows / (double)g->V : 0.0;
  info->device_bytes = g->bytes;
  info->gather_tiles = g->plan.nchunks;
  info->table_vertices = g->plan.tab_cap;
  info->staged_segments = g->plan.m;
  info->staged_edges = g->plan.m > 0 ? g->edge_base[g->plan.m] : 0;
  info->ctas_per_sm = g->plan.ctas_per_sm;
  info->gather_threads = g->plan.threads;
  info->gather_overlap = g->plan.overlap;
  info->affine_segments = g->plan.m2 - g->plan.m;
  info->affine_edges = g->plan.m2 > g->plan.m ? g->edge_base[g->plan.m2] - g->edge_base[g->plan.m]
                                              : 0;
  return CG_OK;
}

int cg_segmented_stats(const cg_segmented* g, int64_t* q_rows_total, double* q,
                       size_t* device_bytes) {
  CG_ARG(g != nullptr, "cg_segmented_stats: null handle");
  if (q_rows_total) *q_rows_total = g->rows;
  if (q) *q = g->V ? (double)g->rows / (double)g->V : 0.0;
  if (device_bytes) *device_bytes = (size_t)g->bytes;
  return CG_OK;
}

int pr_set_gather_config(cg_segmented* g, int32_t threads, int32_t ctas_per_sm,
                         int32_t table_vertices, cudaStream_t stream) {
  CG_ARG(g != nullptr, "pr_set_gather_config: null handle");
  CG_ARG(table_vertices >= -1, "pr_set_gather_config: table_vertices must be >= -1");
  const int t = g->plan.threads, c = g->plan.ctas_per_sm, tab = g->plan.table_request;
  const int rc = seg_plan_configure(&g->plan, threads, ctas_per_sm, table_vertices, stream);
  if (!g->plan.ready)  // it failed half way (memory): back to the previous one, if that goes
    seg_plan_configure(&g->plan, t, c, tab, stream);
  return rc;
}

int pr_set_gather_overlap(cg_segmented* g, int32_t cached_warps, cudaStream_t stream) {
  CG_ARG(g != nullptr, "pr_set_gather_overlap: null handle");
  CG_ARG(cached_warps >= 0 && cached_warps <= 24,
         "pr_set_gather_overlap: cached_warps must be in [0, 24] (got %d)", cached_warps);
  const int before = g->plan.overlap_request;
  g->plan.overlap_request = cached_warps;
  const int rc = seg_plan_configure(&g->plan, g->plan.threads, g->plan.ctas_per_sm,
                                    g->plan.table_request, stream);
  if (rc != CG_OK) {  // keep the previous, valid configuration
    g->plan.overlap_request = before;
    seg_plan_configure(&g->plan, g->plan.threads, g->plan.ctas_per_sm, g->plan.table_request,
                       stream);
  }
  return rc;
}

int pr_set_gather_affine(cg_segmented* g, double head_min_avg_degree, cudaStream_t stream) {
  CG_ARG(g != nullptr, "pr_set_gather_affine: null handle");
  CG_ARG(head_min_avg_degree >= 0.0, "pr_set_gather_affine: head_min_avg_degree must be >= 0");
  const double before = g->plan.affine_head;
  g->plan.affine_head = head_min_avg_degree;
  const int rc = seg_plan_configure(&g->plan, g->plan.threads, g->plan.ctas_per_sm,
                                    g->plan.table_request, stream);
  if (rc != CG_OK) {  // keep the previous, valid configuration
    g->plan.affine_head = before;
    seg_plan_configure(&g->plan, g->plan.threads, g->plan.ctas_per_sm, g->plan.table_request,
                       stream);
  }
  return rc;
}

int pr_gather_table_capacity(int32_t ctas_per_sm) { return seg_table_capacity(ctas_per_sm); }

int pr_plan_bounds(const int32_t* dev_outdeg, int32_t V, int32_t smem_vertices,
                   double min_avg_degree, int32_t max_global_vertices, int32_t k_max,
                   int64_t* host_bounds, int32_t* k_out, cudaStream_t stream) {
  CG_ARG(dev_outdeg && host_bounds && k_out && V >= 1, "pr_plan_bounds: bad arguments");
  CG_ARG(k_max >= 1 && k_max <= kMaxSegments, "pr_plan_bounds: k_max must be in [1, %d]",
         kMaxSegments);
  if (max_global_vertices <= 0) {  // half of this GPU's L2 in 4-byte source values
    DeviceInfo di{};
    CG_TRY(device_info(&di));
    max_global_vertices = (int32_t)std::max<int64_t>(
        1, std::min<int64_t>((int64_t)(di.l2_bytes / 8), (int64_t)0x7FFFFFFF));
  }
  if (smem_vertices < 0) smem_vertices = seg_table_capacity(1);
  // the out-edges of each table-sized range, and the end of the sources that have
  // any: on the device (copying the degrees to the host and adding them there took 4
  // ms of a 4 M-vertex graph's 21 ms from CSR to ranks), but from a copy of the
  // degrees where these are few: scratch and a kernel take 31 us, but 80 where the
  // pool has given its memory back (3,000 vertices from a copy 23 us, 30,000 33, 65,536
  // 47)
  const int64_t nr = smem_vertices > 0 ? std::min<int64_t>(ceil_div(V, smem_vertices), k_max) : 0;
  std::vector<int64_t> sums(nr + 1, 0);
  if (V <= kFewDegrees) {
    std::vector<int32_t> deg(V);
    CG_CUDA(cudaMemcpyAsync(deg.data(), dev_outdeg, sizeof(int32_t) * (size_t)V,
                            cudaMemcpyDeviceToHost, stream));
    CG_CUDA(cudaStreamSynchronize(stream));
    for (int64_t q = 0; q < nr; ++q)
      sums[q] = std::accumulate(deg.begin() + q * smem_vertices,
                                deg.begin() + std::min<int64_t>(V, (q + 1) * smem_vertices),
                                (int64_t)0);
    for (sums[nr] = V; sums[nr] > 0 && deg[sums[nr] - 1] == 0;) --sums[nr];
  } else {
    Scratch tmp(stream);
    int64_t* d = nullptr;
    CG_CUDA(tmp.get(&d, nr + 1));
    CG_CUDA(cudaMemsetAsync(d, 0, sizeof(int64_t) * (size_t)(nr + 1), stream));
    range_degree_kernel<<<grid_for(V, 256), 256, 0, stream>>>(
        dev_outdeg, V, std::max(smem_vertices, 1), nr, d);
    CG_LAUNCH_CHECK();
    CG_CUDA(cudaMemcpyAsync(sums.data(), d, sizeof(int64_t) * (size_t)(nr + 1),
                            cudaMemcpyDeviceToHost, stream));
    CG_CUDA(cudaStreamSynchronize(stream));
  }
  std::vector<int64_t> b = {0};
  int64_t lo = 0;
  if (smem_vertices > 0) {
    while (lo < V && (int)b.size() < k_max) {
      const int64_t n = std::min<int64_t>(smem_vertices, V - lo);
      if ((double)sums[lo / smem_vertices] < min_avg_degree * (double)n) break;
      lo += n;
      b.push_back(lo);
    }
  }
  if (lo < V) {
    // sources without out-edges at the end of the range (all of them, after
    // clustering) form one segment of their own: it has no edges to cut
    const int64_t end = std::max(lo, sums[nr]);
    const int64_t left_k = k_max - ((int64_t)b.size() - 1) - (end < V && end > lo ? 1 : 0);
    if (left_k < 1) {
      // no room: the last shared-memory segment absorbs the rest
      if (b.size() > 1)
        b.back() = V;
      else
        b.push_back(V);  // (there is none)
    } else {
      if (end > lo) {
        int64_t parts = std::max<int64_t>(1, ceil_div(end - lo, max_global_vertices));
        if (parts > left_k) parts = left_k;
        const int64_t step = ceil_div(end - lo, parts);
        for (int64_t q = 1; q <= parts; ++q) b.push_back(std::min<int64_t>(end, lo + q * step));
      }
      if (b.back() < V) b.push_back(V);
    }
  }
  *k_out = (int32_t)(b.size() - 1);
  for (size_t q = 0; q < b.size(); ++q) host_bounds[q] = b[q];
  return CG_OK;
}

int cg_segmented_export(const cg_segmented* g, int64_t* h_bounds, int64_t* h_row_base,
                        int64_t* h_edge_base, int64_t* d_row_ptr, int32_t* d_col,
                        int32_t* d_idx_map, int32_t* d_block_start, cudaStream_t s) {
  CG_ARG(g != nullptr, "cg_segmented_export: null handle");
  for (int q = 0; q <= g->k; ++q) {
    if (h_bounds) h_bounds[q] = g->bounds[q];
    if (h_row_base) h_row_base[q] = g->row_base[q];
    if (h_edge_base) h_edge_base[q] = g->edge_base[q];
  }
  if (d_row_ptr) {
    to_i64_kernel<<<grid_for(g->rows + 1, 256), 256, 0, s>>>(g->row_ptr, g->rows + 1, d_row_ptr);
    CG_LAUNCH_CHECK();
  }
  if (d_col && g->E > 0) CG_TRY(seg_plan_export_col(g->plan, g->row_ptr, d_col, s));
  if (d_idx_map && g->rows > 0)
    CG_CUDA(cudaMemcpyAsync(d_idx_map, g->idx_map, sizeof(int32_t) * g->rows,
                            cudaMemcpyDeviceToDevice, s));
  if (d_block_start) {
    int64_t* d_rb = nullptr;
    CG_CUDA(cudaMallocAsync((void**)&d_rb, sizeof(int64_t) * (g->k + 1), s));
    cudaError_t e = cudaMemcpyAsync(d_rb, g->row_base.data(), sizeof(int64_t) * (g->k + 1),
                                    cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) {
      blk_local_kernel<<<grid_for((int64_t)g->k * (g->nb + 1), 256), 256, 0, s>>>(
          g->idx_map, d_rb, g->k, g->B, g->nb, d_block_start);
      e = cudaGetLastError();
    }
    cudaFreeAsync(d_rb, s);
    if (e != cudaSuccess) return cuda_fail(e, "cg_segmented_export", __FILE__, __LINE__);
  }
  CG_CUDA(cudaStreamSynchronize(s));
  return CG_OK;
}

int cg_segmented_destroy(cg_segmented* g) {
  if (!g) return CG_OK;
  int cur = 0;
  const int dev = g->device;
  cudaGetDevice(&cur);
  if (cur != dev) cudaSetDevice(dev);
  cudaDeviceSynchronize();
  free_segmented(g);
  delete g;
  if (cur != dev) cudaSetDevice(cur);
  return CG_OK;
}

}  // extern "C"
