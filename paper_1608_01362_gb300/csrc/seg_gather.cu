// Flagged-edge segment gather: plan construction and the kernel.
#include <algorithm>

#include "carry_runs.cuh"
#include "ranges.cuh"
#include "staged_stream.cuh"

namespace cg {
namespace {

__device__ __forceinline__ int last_le(const int64_t* a, int n, int64_t v) {
  // last index q in [0, n) with a[q] <= v (a ascending, a[0] <= v)
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] <= v) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

__global__ void export_col_kernel(const uint32_t* __restrict__ colf,
                                  const int32_t* __restrict__ rp, int64_t rows,
                                  const int64_t* __restrict__ row_base,
                                  const int64_t* __restrict__ edge_base,
                                  const int64_t* __restrict__ cstart,
                                  const int64_t* __restrict__ bounds, int k,
                                  int32_t* __restrict__ col) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; i < rows; i += nw) {
    const int s = last_le(row_base, k + 1, i);
    const int64_t shift = cstart[s] - edge_base[s];
    const int32_t src0 = (int32_t)bounds[s];
    for (int64_t e = rp[i] + lane; e < rp[i + 1]; e += 32)
      col[e] = src0 + (int32_t)(colf[e + shift] & ~kRowEndFlag);
  }
}

// The row open at each chunk's end (-1 when the chunk ends a row): the
// subgraph row of the chunk's last edge, if that row continues past it.
__global__ void open_row_kernel(const int32_t* __restrict__ rp,
                                const int64_t* __restrict__ row_base,
                                const int64_t* __restrict__ edge_base,
                                const int64_t* __restrict__ chunk_base, int k, int64_t size,
                                int64_t nchunks, int32_t* __restrict__ open_row) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int s = last_le(chunk_base, k + 1, c);
    const int64_t e0 = edge_base[s] + (c - chunk_base[s]) * size;
    const int64_t e = min(e0 + size, edge_base[s + 1]) - 1;  // the chunk's last edge
    int64_t lo = row_base[s], hi = row_base[s + 1];  // last row with rp[row] <= e
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (rp[mid] <= e) lo = mid + 1; else hi = mid;
    }
    open_row[c] = (int64_t)rp[lo] - 1 > e ? (int32_t)(lo - 1) : -1;
  }
}

template <class Op, bool TILES>
__global__ void __launch_bounds__(256)
seg_fixup_kernel(const int32_t* carry_row, const typename Op::T* carry, int64_t n,
                 typename Op::T* out, const typename Op::T* tiles) {
  if (!chain_begin()) return;
  fix_runs<Op, TILES>(carry_row, carry, n, out, tiles);
}

template <class Op>
__global__ void __launch_bounds__(256)
carry_tiles_kernel(const int32_t* carry_row, const typename Op::T* carry, int64_t n,
                   typename Op::T* tiles) {
  if (!chain_begin()) return;
  carry_tile_sums<Op>(carry_row, carry, n, tiles);
}

// Does a row have all of kLongRun aligned carries?
__global__ void long_runs_kernel(const int32_t* __restrict__ carry_row, int64_t n,
                                 unsigned* __restrict__ found) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n / kLongRun;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int32_t r = carry_row[t * kLongRun];
    if (r >= 0 && carry_row[(t + 1) * kLongRun - 1] == r) *found = 1u;
  }
}

// Subgraph row of each chunk's first edge (chunks of `size` edges; the staged
// segments have none).
__global__ void first_row_kernel(const int32_t* __restrict__ rp,
                                 const int64_t* __restrict__ row_base,
                                 const int64_t* __restrict__ edge_base,
                                 const int64_t* __restrict__ chunk_base, int k, int64_t size,
                                 int64_t nchunks, int32_t* __restrict__ first_row) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int s = last_le(chunk_base, k + 1, c);
    const int64_t e = edge_base[s] + (c - chunk_base[s]) * size;
    int64_t lo = row_base[s], hi = row_base[s + 1];  // last row with rp[row] <= e
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (rp[mid] <= e) lo = mid + 1; else hi = mid;
    }
    first_row[c] = (int32_t)(lo - 1);
  }
}

// One L1/L2 chunk: segment-local chunk j (global chunk c) of 32 * IPL edges of a
// segment whose sources start at lo; lane l holds edges [IPL l, IPL (l + 1)).
// Eight edges per lane, or four where there are few edges: chunks are then few
// per warp, and a launch is a chain of two of them.  The line lies between the
// largest size at which four were faster and the smallest at which eight were (0.3
// M edges 10.3 -> 8.1 us with four, 3.1 M 18.0 -> 16.3, 8.8 M 41.9 -> 40.0, 13.4 M
// 60.3 -> 57.6, 22 M 89.0 -> 91.0, 66 M 260 -> 268).
constexpr int64_t kFewCachedEdges = (int64_t)1 << 24;

template <class Op, int IPL>
__device__ __forceinline__ void cached_chunk(const uint32_t* colf,
                                             const typename Op::T* x, int32_t nx,
                                             int32_t lo, int32_t Es, int32_t cstart, int32_t j,
                                             int32_t c, int32_t frow,
                                             typename Op::T* __restrict__ out,
                                             typename Op::T* __restrict__ carry) {
  using T = typename Op::T;
  constexpr int CHUNK = 32 * IPL;
  const int lane = threadIdx.x & 31;
  const int32_t e0 = j * CHUNK;
  const int n = Es - e0 < CHUNK ? Es - e0 : CHUNK;

  // 1. this lane's edges (16-byte streaming loads; colf is padded)
  const uint4* p = reinterpret_cast<const uint4*>(colf + cstart + e0 + lane * IPL);
  uint32_t cf[IPL];
#pragma unroll
  for (int u = 0; u < IPL; u += 4) {
    const uint4 q = __ldcs(p + u / 4);
    cf[u] = q.x; cf[u + 1] = q.y; cf[u + 2] = q.z; cf[u + 3] = q.w;
  }
  T v[IPL];
  uint32_t fl = 0;
  const int nl = n - lane * IPL;  // valid edges of this lane
#pragma unroll
  for (int u = 0; u < IPL; ++u) {
    const bool ok = u < nl;
    const int32_t src = lo + (int32_t)(cf[u] & ~kRowEndFlag);
    if (ok) fl |= (cf[u] >> 31) << u;
    v[u] = (ok && (uint32_t)src < (uint32_t)nx) ? __ldca(x + src) : Op::identity();
  }

  // 2. rows ended before this lane (exclusive warp prefix of flag counts)
  const int F = __popc(fl);
  int incl = F;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += y;
  }
  const int32_t row0 = frow + (incl - F);

  // 3. sequential fold; rows that start and end in this lane are final
  T acc = Op::identity(), first_val = Op::identity();
  int nf = 0;
#pragma unroll
  for (int u = 0; u < IPL; ++u) {
    acc = Op::op(acc, v[u]);
    if (fl & (1u << u)) {
      if (nf == 0)
        first_val = acc;
      else
        out[row0 + nf] = acc;
      ++nf;
      acc = Op::identity();
    }
  }

  // 4. segmented scan of the open-row parts; completes each lane's first row
  T S = acc;
  int h = F > 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const T y = __shfl_up_sync(0xffffffffu, S, o);
    const int g = __shfl_up_sync(0xffffffffu, h, o);
    if (lane >= o) {
      if (!h) S = Op::op(y, S);
      h |= g;
    }
  }
  const T P = __shfl_up_sync(0xffffffffu, S, 1);
  if (F > 0) out[row0] = lane > 0 ? Op::op(P, first_val) : first_val;

  // 5. the row open at the chunk's end (completed by the carry pieces)
  const uint32_t lf = __shfl_sync(0xffffffffu, fl, (n - 1) / IPL);
  if (lane == 31 && !((lf >> ((n - 1) % IPL)) & 1u)) carry[c] = S;
}

// The L1/L2 launch: every read of a segment in [ct_begin, ct_end) goes
// through L1/L2.  Blocks take block-groups round-robin (the grid sweeps the
// groups in order, which balances blocks when the cost per group varies).
template <class Op, int THREADS, int IPL>
__global__ void __launch_bounds__(THREADS, 2048 / THREADS)
seg_gather_kernel(const uint32_t* colf, const typename Op::T* x,
                  int32_t nx, const int32_t* first_row,
                  const int64_t* seg_cstart, const int32_t* seg_E,
                  const int64_t* seg_chunk, const int32_t* seg_ctile,
                  const int32_t* seg_lo, int k, int32_t ct_begin, int32_t ct_end,
                  typename Op::T* out, typename Op::T* carry) {
  constexpr int WARPS = THREADS / 32;
  if (!chain_begin()) return;
  const int w = threadIdx.x >> 5;
  const int32_t my_lo = ct_begin + (int32_t)blockIdx.x;
  const int32_t step = (int32_t)gridDim.x;
  if (my_lo >= ct_end) return;
  int s;  // segment of the first group; later ones are found by stepping forward
  {
    int a = 0, b = k + 1;
    while (a < b) {
      const int mid = (a + b) >> 1;
      if (seg_ctile[mid] <= my_lo) a = mid + 1; else b = mid;
    }
    s = a - 1;
  }
  int32_t lo = 0, Es = 0, cstart = 0, cbase = 0, ctbase = 0, ctnext = -1;

  for (int32_t ct = my_lo; ct < ct_end; ct += step) {
    if (ct >= ctnext) {
      while (ct >= seg_ctile[s + 1]) ++s;
      lo = seg_lo[s];
      Es = seg_E[s];
      cstart = (int32_t)seg_cstart[s];
      cbase = (int32_t)seg_chunk[s];
      ctbase = seg_ctile[s];
      ctnext = seg_ctile[s + 1];
    }
    const int32_t j = (ct - ctbase) * WARPS + w;  // chunk of this warp within the segment
    if (j * 32 * IPL >= Es) continue;             // warp-uniform
    cached_chunk<Op, IPL>(colf, x, nx, lo, Es, cstart, j, cbase + j, first_row[cbase + j], out,
                     carry);
  }
}

// Copy n values into shared memory by threads [0, nt): 16-byte asynchronous
// copies where the source is 16-byte aligned (all of a thread's copies are in
// flight at once and pass no register), 4-byte ones otherwise.  The caller's
// next barrier publishes the table.
template <typename T>
__device__ __forceinline__ void stage_table(const T* src, int n, T* dst, int tid,
                                            int nt) {
  static_assert(sizeof(T) == 4, "4-byte values");
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const int n4 = (reinterpret_cast<uintptr_t>(src) & 15) == 0 ? n >> 2 : 0;
  for (int i = tid; i < n4; i += nt)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(d + 16 * i),
                 "l"(src + 4 * i)
                 : "memory");
  for (int i = (n4 << 2) + tid; i < n; i += nt)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(d + 4 * i), "l"(src + i)
                 : "memory");
  asm volatile("cp.async.wait_all;" ::: "memory");
}

// The staged segments [0, m) and their tasks' shares among the blocks.
struct StagedShare {
  RangeShare ranges;
  unsigned* done;           // blocks finished
  const int32_t* seg_lo;
  const int32_t* seg_tab;
  int m;
};

// The staged schedule, run by threads [0, nt) of a block: segments [0, m)
// are read from a shared-memory copy of their source values.  A block works
// through its own range of tasks, which meets one or two segments, and then
// helps with the fullest range (ranges.cuh).  (The earlier schedule handed out
// small pieces of all the tasks in order, so every block met nearly every
// segment: 31 table copies per block on RMAT-25, each as long as 1.8 us of L2
// reads at 64 bytes per cycle and SM, and two barriers per piece.)
template <class Op>
__device__ __forceinline__ void staged_pieces(
    const StagedTasks& q, const StagedShare& sh, const typename Op::T* x,
    typename Op::T* __restrict__ out, typename Op::T* __restrict__ carry, typename Op::T* tab,
    int nt, RangeSlots* slots) {
  using T = typename Op::T;
  const int tid = threadIdx.x, w = tid >> 5;
  int s = -1;               // the segment in the table
  int v = (int)blockIdx.x;  // the range being worked on
  if (tid == 0) tab[q.pad] = Op::identity();  // the first table's barrier publishes it
  int32_t t, hi;
  while (next_range(sh.ranges, nt, slots, &v, &t, &hi)) {
    while (t < hi) {
      const int sn = segment_of_task(q.seg_task, sh.m, t);
      const int32_t te = __ldca(q.seg_task + sn + 1);
      if (sn != s) {
        s = sn;
        group_sync(nt);  // every warp is done reading the previous table
        stage_table<T>(x + sh.seg_lo[s], sh.seg_tab[s], tab, tid, nt);
        group_sync(nt);
      }
      const int32_t e = min(hi, te);
      staged_run<Op>(q, t, e, w, nt >> 5, tab, out, carry);
      t = e;
    }
  }
}

// The last block to finish clears the n counters that the launch used, ready
// for the next one (which then needs no memset before it).  Every thread of the
// block calls it, when the block is done with the counters.
__device__ __forceinline__ void counters_done(unsigned* counters, int n, unsigned* done) {
  __shared__ bool s_last;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    s_last = atomicAdd(done, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  for (int i = threadIdx.x; i < n; i += blockDim.x) counters[i] = 0u;
  if (threadIdx.x == 0) *done = 0u;
}

// The staged launch: every thread of the block runs the staged schedule.
template <class Op, int THREADS>
__global__ void __launch_bounds__(THREADS, 1024 / THREADS)
staged_gather_kernel(StagedTasks q, StagedShare sh, const typename Op::T* x,
                     typename Op::T* out, typename Op::T* carry) {
  using T = typename Op::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RangeSlots slots;
  if (!chain_begin()) return;
  staged_pieces<Op>(q, sh, x, out, carry, reinterpret_cast<T*>(smem_raw), THREADS, &slots);
  counters_done(sh.ranges.next, (int)gridDim.x, sh.done);
}

// The segment-affine staged launch (the nested form of two-level segmenting:
// the cold part of the source range, which an L2-sized segment would serve
// with random L2 reads, cut into shared-memory-sized segments).  Each block
// takes whole segments of [m, m2) from a counter, in order (heaviest first
// after clustering), stages the segment's table once and streams all its
// tasks with every warp; low-degree segments thus pay one table copy each
// instead of one per block.
template <class Op>
__global__ void __launch_bounds__(1024, 1)
affine_gather_kernel(StagedTasks q, const typename Op::T* x,
                     const int32_t* seg_lo, const int32_t* seg_tab,
                     int m, int m2, unsigned* next_seg, unsigned* done,
                     typename Op::T* out, typename Op::T* carry) {
  using T = typename Op::T;
  if (!chain_begin()) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  T* tab = reinterpret_cast<T*>(smem_raw);
  __shared__ int32_t s_seg;
  const int tid = threadIdx.x, w = tid >> 5;
  if (tid == 0) tab[q.pad] = Op::identity();
  for (;;) {
    __syncthreads();  // every warp is done with the previous table and s_seg
    if (tid == 0) s_seg = m + (int32_t)atomicAdd(next_seg, 1u);
    __syncthreads();
    const int s = s_seg;
    if (s >= m2) break;
    const int32_t tb = q.seg_task[s], te = q.seg_task[s + 1];
    if (tb == te) continue;
    stage_table<T>(x + seg_lo[s], seg_tab[s], tab, tid, 1024);
    __syncthreads();
    staged_run<Op>(q, tb, te, w, 32, tab, out, carry);
  }
  counters_done(next_seg, 1, done);
}

// L1/L2 chunks of segments [m, k) taken from a queue (a global counter of chunks,
// kCachedGrab at a time): a warp's successive grabs only move forward, so its segment
// is found by stepping.  Two at a time: with one the counter and the search cost (4
// M vertices, 8 warps per block: 128 us, 119 so), with four the last grabs outlast
// the rest (0.5 M, 4 warps: 40 us, 30 so).  Pulling a grab's edges into L2 when it is
// taken was of no use (33 M, 2 warps: 1051 us with, 1014 without).
constexpr int kCachedGrab = 2;

template <class Op, int IPL>
__device__ __forceinline__ void cached_queue(
    const uint32_t* colf, const typename Op::T* x, int32_t nx,
    const int32_t* first_row, const int64_t* seg_cstart,
    const int32_t* seg_E, const int64_t* seg_chunk,
    const int32_t* seg_lo, int m, int k, unsigned* __restrict__ next_chunk,
    typename Op::T* __restrict__ out, typename Op::T* __restrict__ carry) {
  const int lane = threadIdx.x & 31;
  const int32_t c_begin = (int32_t)seg_chunk[m], c_end = (int32_t)seg_chunk[k];
  int s = m;
  int32_t lo = 0, Es = 0, cstart = 0, cbase = 0, cnext = -1;
  for (;;) {
    int32_t c0 = 0;
    if (lane == 0) c0 = (int32_t)atomicAdd(next_chunk, (unsigned)kCachedGrab);
    c0 = __shfl_sync(0xffffffffu, c0, 0) + c_begin;
    if (c0 >= c_end) break;
    const int32_t c1 = min(c0 + kCachedGrab, c_end);
    for (int32_t c = c0; c < c1; ++c) {
      if (c >= cnext) {
        while (c >= (int32_t)seg_chunk[s + 1]) ++s;
        lo = seg_lo[s];
        Es = seg_E[s];
        cstart = (int32_t)seg_cstart[s];
        cbase = (int32_t)seg_chunk[s];
        cnext = (int32_t)seg_chunk[s + 1];
      }
      cached_chunk<Op, IPL>(colf, x, nx, lo, Es, cstart, c - cbase, c, first_row[c], out, carry);
    }
  }
}

// Both kinds in one launch (one 1024-thread block per SM): threads
// [0, staged_threads) run the staged schedule (named barrier 1 among them),
// the other warps serve the L1/L2 segments from the chunk queue from the
// start, and the staged warps join that queue when their pieces run out.
// The cold segments' random reads go to L2 while the staged warps read
// shared memory, so the two kinds of lookup proceed side by side.
template <class Op, int IPL>
__global__ void __launch_bounds__(1024, 1)
overlap_gather_kernel(StagedTasks q, StagedShare sh, const uint32_t* colf,
                      const typename Op::T* x, int32_t nx,
                      const int32_t* first_row,
                      const int64_t* seg_cstart, const int32_t* seg_E,
                      const int64_t* seg_chunk, const int32_t* seg_lo,
                      int m, int k, int staged_threads, unsigned* next_chunk,
                      typename Op::T* out, typename Op::T* carry) {
  using T = typename Op::T;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ RangeSlots slots;
  if (!chain_begin()) return;
  if ((int)threadIdx.x < staged_threads)
    staged_pieces<Op>(q, sh, x, out, carry, reinterpret_cast<T*>(smem_raw), staged_threads, &slots);
  cached_queue<Op, IPL>(colf, x, nx, first_row, seg_cstart, seg_E, seg_chunk, seg_lo, m, k, next_chunk,
                   out, carry);
  counters_done(next_chunk, 4 + (int)gridDim.x, sh.done);  // the ranges' lie behind it
}

// Block b's first task: equal stretches of the stream (no tasks: empty shares).
__global__ void staged_share_kernel(const uint4* __restrict__ desc, int32_t ntasks, int grid,
                                    int32_t* __restrict__ blk_task) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= grid; b += gridDim.x * blockDim.x) {
    if (ntasks == 0) {
      blk_task[b] = 0;
      continue;
    }
    const uint4 e = desc[ntasks - 1];
    const int64_t total = (int64_t)e.x + (e.y >> 16);
    const int64_t want = total * b / grid;
    int32_t lo = 0, hi = ntasks;
    while (lo < hi) {
      const int32_t mid = (lo + hi) >> 1;
      if ((int64_t)desc[mid].x < want) lo = mid + 1; else hi = mid;
    }
    blk_task[b] = b == grid ? ntasks : lo;
  }
}

}  // namespace

int seg_table_capacity(int ctas) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 0;
  int sm_smem = 0, reserved = 0, optin = 0;
  cudaDeviceGetAttribute(&sm_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (ctas < 1) ctas = 1;
  int64_t per = (int64_t)sm_smem / ctas - reserved;
  if (per > optin) per = optin;
  per -= 128;  // the gather kernels' own static shared memory
  if (per <= 0) return 0;
  return (int)((per / 4) & ~31LL);
}

int seg_plan_alloc(int64_t E, int k, const std::vector<int64_t>& edge_base,
                   const std::vector<int64_t>& src_bounds, SegPlan* p, cudaStream_t s) {
  p->k = k;
  p->E = E;
  p->edge_base = edge_base;
  p->src_bounds = src_bounds;
  p->h_cstart.assign(k + 1, 0);
  for (int q = 0; q < k; ++q) {
    const int64_t Eq = edge_base[q + 1] - edge_base[q];
    p->h_cstart[q + 1] = p->h_cstart[q] + ((Eq + 7) & ~7LL);
  }
  p->colf_len = p->h_cstart[k] + kMaxChunkEdges;  // chunks may read past their segment's end
  CG_CUDA(cudaMalloc((void**)&p->colf, sizeof(uint32_t) * p->colf_len));
  // The segments' arrays, one allocation and one upload: meta (row_base, which
  // the caller's build writes, edge_base, cstart, bounds), then seg_E and
  // seg_lo; behind them what seg_plan_configure uploads in its turn (seg_chunk,
  // seg_ctile, seg_tab), and the staged launch's counters and shares.
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  const size_t n = (size_t)k + 1, most = (size_t)di.sm_count * 2;  // blocks of any staged shape
  const size_t words = 2 * 4 * n + 2 * n + 2 * n + 3 * n + (4 + most) + (most + 1) + 1;
  CG_CUDA(cudaMalloc((void**)&p->meta, 4 * words));
  int32_t* w = reinterpret_cast<int32_t*>(p->meta) + 2 * 4 * n;
  p->seg_cstart = p->meta + 2 * n;
  p->seg_E = w;
  p->seg_lo = w + n;
  w += 2 * n;  // 8-byte aligned: an even number of words before it
  p->seg_chunk = reinterpret_cast<int64_t*>(w);
  p->seg_ctile = w + 2 * n;
  p->seg_tab = w + 3 * n;
  p->seg_task = w + 4 * n;
  p->counter = reinterpret_cast<unsigned*>(w + 5 * n);
  p->blk_task = w + 5 * n + 4 + most;
  p->found = reinterpret_cast<unsigned*>(p->blk_task + most + 1);
  CG_CUDA(cudaMemsetAsync(p->counter, 0, 4 * ((4 + most) + (most + 1)), s));  // and the shares
  std::vector<int64_t> up(4 * n, 0);  // edge_base, cstart, bounds, then seg_E and seg_lo
  int32_t* eo = reinterpret_cast<int32_t*>(up.data() + 3 * n);
  for (size_t q = 0; q < n; ++q) {
    up[q] = edge_base[q];
    up[n + q] = p->h_cstart[q];
    up[2 * n + q] = src_bounds[q];
    eo[q] = q + 1 < n ? (int32_t)(edge_base[q + 1] - edge_base[q]) : 0;
    eo[n + q] = (int32_t)src_bounds[q];
  }
  // (a copy from pageable memory returns once the source has been read)
  CG_CUDA(cudaMemcpyAsync(p->meta + n, up.data(), sizeof(int64_t) * up.size(),
                          cudaMemcpyHostToDevice, s));
  return CG_OK;
}

int seg_plan_finish(SegPlan* p, const int32_t* rp32, int64_t rows,
                    const std::vector<int64_t>& row_base, cudaStream_t s) {
  p->rows = rows;
  p->rp32 = rp32;
  p->row_base = row_base;
  return seg_plan_configure(p, 1024, 1, -1, s);
}

// The staged kernels may take the largest table (a launch asks for its own).
template <class Op>
static int allow_tables() {
  const void* fns[] = {(const void*)staged_gather_kernel<Op, 1024>,
                       (const void*)staged_gather_kernel<Op, 512>,
                       (const void*)affine_gather_kernel<Op>,
                       (const void*)overlap_gather_kernel<Op, 4>,
                       (const void*)overlap_gather_kernel<Op, 8>};
  const int most = 4 * seg_table_capacity(1) + 16;
  for (const void* f : fns)
    CG_CUDA(cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  return CG_OK;
}

// The staged segments' tasks, the L1/L2 segments' chunks and the carries of both.
static int layout(SegPlan* p, int m2, int pad, int chunk_edges, const std::vector<int64_t>& chunk,
                  const std::vector<int32_t>& ctile, const std::vector<int32_t>& tn,
                  cudaStream_t s) {
  const int k = p->k;
  const int64_t ncached = chunk[k];
  // the carries of the staged rows' full pieces follow the chunks'
  CG_TRY(staged_build(p, m2, pad, ncached, s));
  // seg_chunk, seg_ctile, seg_tab lie one behind the other
  const size_t n = (size_t)k + 1;
  std::vector<int32_t> up(4 * n, 0);
  std::copy(chunk.begin(), chunk.end(), reinterpret_cast<int64_t*>(up.data()));
  std::copy(ctile.begin(), ctile.end(), up.begin() + 2 * n);
  std::copy(tn.begin(), tn.begin() + k, up.begin() + 3 * n);
  CG_CUDA(cudaMemcpyAsync(p->seg_chunk, up.data(), sizeof(int32_t) * up.size(),
                          cudaMemcpyHostToDevice, s));
  if (ncached > 0) {
    first_row_kernel<<<grid_for(ncached, 256), 256, 0, s>>>(
        p->rp32, p->meta, p->meta + (k + 1), p->seg_chunk, k, chunk_edges, ncached, p->first_row);
    CG_LAUNCH_CHECK();
    open_row_kernel<<<grid_for(ncached, 256), 256, 0, s>>>(
        p->rp32, p->meta, p->meta + (k + 1), p->seg_chunk, k, chunk_edges, ncached,
        p->carry_row);
    CG_LAUNCH_CHECK();
  }
  unsigned long_runs = 0;
  if (p->ncarry >= kLongRun) {
    CG_CUDA(cudaMemsetAsync(p->found, 0, sizeof(unsigned), s));
    long_runs_kernel<<<grid_for(p->ncarry / kLongRun, 256), 256, 0, s>>>(p->carry_row, p->ncarry,
                                                                         p->found);
    CG_LAUNCH_CHECK();
    CG_CUDA(cudaMemcpyAsync(&long_runs, p->found, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    CG_CUDA(cudaStreamSynchronize(s));
  }
  p->long_runs = long_runs != 0;
  return CG_OK;
}

int seg_plan_configure(SegPlan* p, int threads, int ctas_per_sm, int tab_vertices,
                       cudaStream_t s) {
  CG_TRY(allow_tables<SumF32>());
  CG_TRY(allow_tables<MinI32>());
  if (threads != 512 && threads != 1024) {
    set_error("gather threads must be 512 or 1024 (got %d)", threads);
    return CG_ERR_INVALID_ARG;
  }
  const int max_ctas = 1024 / threads;  // the staged kernel holds 64 registers per thread
  if (ctas_per_sm < 1 || ctas_per_sm > max_ctas) {
    set_error("ctas_per_sm must be in [1, %d] for %d threads", max_ctas, threads);
    return CG_ERR_INVALID_ARG;
  }
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  const int cap = seg_table_capacity(ctas_per_sm);
  int tab = tab_vertices < 0 ? cap : std::min(tab_vertices, cap);
  // staged sources are 16-bit segment-local indices, one of them the identity's
  tab = std::min(tab, 65532) & ~3;
  const int k = p->k;
  // staged prefix: leading segments that fit the table and carry enough
  // edges (>= 4 per source) for staging them in shared memory to pay
  // (with the segment-affine plan: >= affine_head edges per source, the
  // rest of the table-sized segments go one block per segment)
  const double head_deg = p->affine_head > 0.0 ? std::max(4.0, p->affine_head) : 4.0;
  int m = 0;
  int64_t tabmax = 0;
  while (m < k && tab > 0) {
    const int64_t size = p->src_bounds[m + 1] - p->src_bounds[m];
    const int64_t Eq = p->edge_base[m + 1] - p->edge_base[m];
    if (size > tab || (double)Eq < head_deg * (double)size) break;
    tabmax = std::max(tabmax, size);
    ++m;
  }
  // segment-affine staged segments [m, m2): the table-sized segments after the
  // head, when asked for (each one's table is staged once, by one block)
  int m2 = m;
  if (p->affine_head > 0.0) {
    if (threads != 1024 || ctas_per_sm != 1) {
      set_error("segment-affine staging needs 1024 threads and 1 block per SM (got %d x %d)",
                threads, ctas_per_sm);
      return CG_ERR_INVALID_ARG;
    }
    if (p->overlap_request > 0) {
      set_error("segment-affine staging and the overlapped gather exclude each other");
      return CG_ERR_INVALID_ARG;
    }
    while (m2 < k && tab > 0 && p->src_bounds[m2 + 1] - p->src_bounds[m2] <= tab) {
      tabmax = std::max(tabmax, p->src_bounds[m2 + 1] - p->src_bounds[m2]);
      ++m2;
    }
  }
  // one overlapped launch needs the 1024 x 1 shape
  if (p->overlap_request > 0 && (threads != 1024 || ctas_per_sm != 1)) {
    set_error("gather overlap needs 1024 threads and 1 block per SM (got %d x %d)", threads,
              ctas_per_sm);
    return CG_ERR_INVALID_ARG;
  }
  const int warps_b = 1024 / 32;
  const int tab_cap = (int)((tabmax + 3) & ~3LL);
  // chunks of the segments read through L1/L2
  int64_t cached = 0;
  for (int q = m2; q < k; ++q) cached += p->edge_base[q + 1] - p->edge_base[q];
  const int cached_ipl = cached < kFewCachedEdges ? 4 : 8, chunk_edges = 32 * cached_ipl;
  std::vector<int64_t> chunk(k + 1, 0);
  std::vector<int32_t> ctile(k + 1, 0), tn(k > 0 ? k : 1, 0);
  for (int q = 0; q < k; ++q) {
    chunk[q + 1] =
        chunk[q] + (q < m2 ? 0 : ceil_div(p->edge_base[q + 1] - p->edge_base[q], chunk_edges));
    tn[q] = q < m2 ? (int32_t)(p->src_bounds[q + 1] - p->src_bounds[q]) : 0;
  }
  const int64_t ncached = chunk[k];
  for (int q = 0; q < k; ++q)  // block-groups of the L1/L2 launch
    ctile[q + 1] = ctile[q] + (int32_t)ceil_div(chunk[q + 1] - chunk[q], warps_b);
  // tasks, chunks and carries stay where they come out as they are (another shape or
  // overlap with the same segments staged)
  const bool same = p->ready && p->m2 == m2 && p->tab_cap == tab_cap &&
                    p->cached_ipl == cached_ipl && p->ncached == ncached;
  p->ready = false;
  if (!same) CG_TRY(layout(p, m2, tab_cap, chunk_edges, chunk, ctile, tn, s));
  p->cached_ipl = cached_ipl;
  p->ncached = ncached;
  p->threads = threads;
  p->ctas_per_sm = ctas_per_sm;
  p->tab_cap = tab_cap;
  p->table_request = tab;
  p->m = m;
  p->m2 = m2;
  p->grid_affine = di.sm_count;
  p->nchunks = p->h_seg_task[k] + ncached;
  p->n_ctiles = ctile[k];
  // the staged launch: one block per resident slot, or per task where there are fewer
  // (every SM serves the L1/L2 queue too in an overlapped launch)
  const int32_t head = p->h_seg_task[m];
  // one overlapped launch needs tasks of both kinds (staged segments can all be
  // empty: they have no tasks, and the blocks no shares)
  p->overlap = (head > 0 && cached > 0) ? p->overlap_request : 0;
  p->grid = (int)std::max<int64_t>(1, std::min<int64_t>(head, (int64_t)di.sm_count * ctas_per_sm));
  if (p->overlap > 0) p->grid = di.sm_count;
  p->head_tasks = head;
  staged_share_kernel<<<grid_for(p->grid + 1, 128), 128, 0, s>>>(p->desc, head, p->grid,
                                                                 p->blk_task);
  CG_LAUNCH_CHECK();
  p->grid_l2 = (int)std::max<int64_t>(
      1, std::min<int64_t>(p->n_ctiles, (int64_t)di.sm_count * 2));
  CG_CUDA(cudaStreamSynchronize(s));
  p->ready = true;
  return CG_OK;
}

int seg_plan_carries(SegPlan* p, int64_t n) {
  p->ncarry = n;
  if (n <= p->carry_cap) return CG_OK;
  cudaFree(p->first_row);
  p->first_row = nullptr;
  p->carry_cap = 0;
  CG_CUDA(cudaMalloc((void**)&p->first_row, sizeof(int32_t) * (size_t)(3 * n + n / kCarryTile)));
  p->carry_row = p->first_row + n;
  p->carry = p->first_row + 2 * n;
  p->carry_tiles = p->first_row + 3 * n;
  p->carry_cap = n;
  return CG_OK;
}

void seg_plan_free(SegPlan* p) {
  cudaFree(p->colf);
  cudaFree(p->desc);
  cudaFree(p->meta);
  cudaFree(p->first_row);
  *p = SegPlan();
}

int64_t seg_plan_bytes(const SegPlan& p) {
  return 4 * p.colf_len + p.cs_cap + 12 * p.carry_cap + 4 * (p.carry_cap / kCarryTile) +
         76 * (int64_t)p.k;
}

int seg_plan_export_col(const SegPlan& p, const int32_t* rp, int32_t* col, cudaStream_t s) {
  if (p.rows == 0) return CG_OK;
  const int k = p.k;
  export_col_kernel<<<grid_for(p.rows * 32, 256, 16), 256, 0, s>>>(
      p.colf, rp, p.rows, p.meta, p.meta + (k + 1), p.meta + 2 * (k + 1), p.meta + 3 * (k + 1), k,
      col);
  CG_LAUNCH_CHECK();
  CG_CUDA(cudaStreamSynchronize(s));
  return CG_OK;
}

static StagedTasks staged_tasks(const SegPlan& p) {
  return StagedTasks{p.cs, p.desc, p.seg_task, p.tab_cap};
}

static StagedShare staged_share(const SegPlan& p) {
  return StagedShare{{p.blk_task, p.counter + 4}, p.counter + 2, p.seg_lo, p.seg_tab, p.m};
}

// the table and, behind it, the identity's entry
static size_t staged_smem(const SegPlan& p) { return 4 * (size_t)p.tab_cap + 16; }

template <class Op, int THREADS>
static int launch_staged(const SegPlan& p, const typename Op::T* x, typename Op::T* out,
                         cudaStream_t s) {
  using T = typename Op::T;
  const size_t smem = staged_smem(p);
  auto fn = staged_gather_kernel<Op, THREADS>;
  return launch_chained(fn, p.grid, THREADS, smem, s, staged_tasks(p), staged_share(p), x, out,
                        reinterpret_cast<T*>(p.carry));
}

template <class Op>
static int launch_overlap(const SegPlan& p, const typename Op::T* x, int32_t nx,
                          typename Op::T* out, cudaStream_t s) {
  using T = typename Op::T;
  const size_t smem = staged_smem(p);
  auto fn = p.cached_ipl == 4 ? overlap_gather_kernel<Op, 4> : overlap_gather_kernel<Op, 8>;
  return launch_chained(fn, p.grid, 1024, smem, s, staged_tasks(p), staged_share(p), p.colf, x, nx,
                        p.first_row, p.seg_cstart, p.seg_E, p.seg_chunk, p.seg_lo, p.m, p.k,
                        1024 - 32 * p.overlap, p.counter, out, reinterpret_cast<T*>(p.carry));
}

template <class Op>
int run_seg_gather(const SegPlan& p, const typename Op::T* x, int32_t nx, typename Op::T* out,
                   cudaStream_t s, int phases) {
  if (!p.ready) {
    set_error("segmented gather: its last configuration failed; configure it again");
    return CG_ERR_UNSUPPORTED;
  }
  if (p.nchunks == 0) return CG_OK;
  using T = typename Op::T;
  if (p.overlap > 0) {  // both kinds in one launch, counted as the staged phase
    if (phases & kPhaseStaged) CG_TRY((launch_overlap<Op>(p, x, nx, out, s)));
    phases &= ~(kPhaseStaged | kPhaseCached);
  }
  // staged segments [0, m): read from a shared-memory copy
  if ((phases & kPhaseStaged) && p.head_tasks > 0) {
    if (p.threads == 1024)
      CG_TRY((launch_staged<Op, 1024>(p, x, out, s)));
    else
      CG_TRY((launch_staged<Op, 512>(p, x, out, s)));
  }
  // the table-sized cold segments, one block per segment
  if ((phases & kPhaseCached) && p.m2 > p.m) {
    const size_t smem = staged_smem(p);
    CG_TRY(launch_chained(affine_gather_kernel<Op>, p.grid_affine, 1024, smem, s, staged_tasks(p),
                          x, p.seg_lo, p.seg_tab, p.m, p.m2, p.counter + 1, p.counter + 3, out,
                          reinterpret_cast<T*>(p.carry)));
  }
  // the rest through L1/L2: no shared memory, so the whole on-chip store is L1
  if ((phases & kPhaseCached) && p.n_ctiles > 0) {
    auto fn = p.cached_ipl == 4 ? seg_gather_kernel<Op, 1024, 4> : seg_gather_kernel<Op, 1024, 8>;
    CG_TRY(launch_chained(fn, p.grid_l2, 1024, 0, s, p.colf, x, nx,
                          p.first_row, p.seg_cstart, p.seg_E, p.seg_chunk, p.seg_ctile, p.seg_lo,
                          p.k, 0, (int32_t)p.n_ctiles, out, reinterpret_cast<T*>(p.carry)));
  }
  if ((phases & kPhaseFixup) && p.ncarry > 0) {
    const T* carry = reinterpret_cast<const T*>(p.carry);
    T* tiles = reinterpret_cast<T*>(p.carry_tiles);
    if (p.long_runs)
      CG_TRY(launch_chained(carry_tiles_kernel<Op>, grid_for(p.ncarry / kCarryTile * 32, 256, 8),
                            256, 0, s, p.carry_row, carry, p.ncarry, tiles));
    auto fn = p.long_runs ? seg_fixup_kernel<Op, true> : seg_fixup_kernel<Op, false>;
    CG_TRY(launch_chained(fn, grid_for(p.ncarry, 256, 8), 256, 0, s, p.carry_row, carry, p.ncarry,
                          out, tiles));
  }
  return CG_OK;
}

template int run_seg_gather<SumF32>(const SegPlan&, const float*, int32_t, float*, cudaStream_t,
                                    int);
template int run_seg_gather<MinI32>(const SegPlan&, const int32_t*, int32_t, int32_t*,
                                    cudaStream_t, int);

}  // namespace cg
