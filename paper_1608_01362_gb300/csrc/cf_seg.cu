// The collaborative-filtering gather with the neighbours' factor rows in shared
// memory: CSR segmenting (Section III) of the rating graph.
//
// A gather reads one factor row per rating.  Served from L2 that is 128 bytes
// of random rows per rating (K = 32), and the L2's random-row rate bounds it:
// 9.9 TB/s measured, 1.28 and 1.59 ms per side for 99 M ratings.  A segment of
// `width` neighbour rows (as many as fit in an SM's shared memory: 1,815 at K =
// 32) is decoded to FP32 into a table once, and its ratings read their rows
// from there at up to 128 bytes per cycle and SM.  What it costs is a partial
// gradient row per (vertex, segment) with ratings, written and summed again by
// the update: about 21 ratings share one on the Netflix shape, so 2 x 128 bytes
// of sequential and row traffic replace 21 x 128 bytes of random reads.
//
// A piece is a run of consecutive ratings of one vertex in one segment, at most
// kCfSegPiece of them.  A warp task holds G = 32 / LANES pieces of one segment,
// LANES lanes each, so a piece's gradient needs no reduction over the warp;
// the pieces of a segment are sorted by length, so the G of a task are about
// equally long.  The ratings themselves stay where the caller keeps them: a
// piece is a place in the caller's arrays, which are read on every sweep.
// Each lane holds 8 of the dimensions.  Where two ratings share a
// 128-byte shared-memory phase (K = 32: four lanes, two 16-byte reads per
// row), odd groups read the row's second half first, so the phase's eight
// lanes fall on all 32 banks.
//
// Measured, 99 M ratings, K = 32, hi + lo: gathers 1.59 + 1.28 -> 1.07 + 1.02 ms,
// updates 0.07 -> 0.29 ms per sweep.  What is left is latency, not a unit: the
// loop alone takes 0.61 ms with its stream, vertex rows and gradient rows taken out
// (shared-memory pipe 47% busy).  On the way: 1024 threads of 64 registers 1.59 ms;
// packed FMAs and one shared-out reduction per four ratings (212 -> 104
// instructions) 1.43; 512 threads with the next task's rows and ratings read
// ahead and the one after it asked into L2 1.07.  The same tasks with the rows
// left to the L1 (48 warps, no table) took 1.45.
#include <algorithm>
#include <vector>

#include "cf_seg.cuh"
#include "cf_store.cuh"
#include "rowwalk.cuh"

namespace cg {
namespace {

constexpr int kCfSegPiece = 128;   // ratings per piece at most
constexpr int kLenBits = 7;        // sort key of a piece: segment, then kCfSegPiece - length
constexpr int kCfSegMost = 1024;   // segments at most
// Where segments pay (whole passes of 10 sweeps against the gather from L2):
//   K = 16   never: a row is 64 bytes, half an L2 line (1.26 M ratings 642 ->
//            675 us, 5.6 M 1504 -> 1520);
//   K = 32   from 600 K ratings on (0.46 M: 659 -> 683 us, 0.83 M: 1134 ->
//            1049, 99 M: 29.8 -> 24.1 ms): fewer leave the blocks, each with a table
//            to copy, without tasks;
//   K = 64   always (0.15 M: 809 -> 591 us, 5.3 M: 3870 -> 3020);
// and with at least kMinRun ratings per run, or gradient rows that stay in half
// of the L2: 41 M ratings in runs of 9 spill theirs to DRAM (12.6 -> 15.6 ms),
// 0.6 M in runs of 9 do not (1358 -> 1117 us).
constexpr int64_t kMinRun = 14, kMinRunInL2 = 3, kMinRatings32 = 600000;

bool segments_pay(int K, int64_t R, int64_t nruns, size_t l2_bytes) {
  if (K == 16 || (K == 32 && R < kMinRatings32)) return false;
  if (R >= kMinRun * nruns) return true;
  return R >= kMinRunInL2 * nruns && 4 * (int64_t)K * nruns <= (int64_t)(l2_bytes / 2);
}

constexpr int kCfSegThreads = 512;  // 128 registers a thread

// lanes per rating and 16-byte reads per lane and row
template <int K> struct CfShape {
  static constexpr int kLanes = K == 64 ? 8 : 4, kReads = 2;
};
int pieces_per_task(int K) { return K == 64 ? 4 : 8; }

typedef unsigned long long u64;

// FP32 pairs (Blackwell's packed FMA): d += a b, both halves
__device__ __forceinline__ void fma2(u64& d, u64 a, u64 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 pair(float a, float b) {
  u64 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float halves(u64 d) {
  float a, b;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(d));
  return a + b;
}

// This group's piece of a task (none at or past `end`).
__device__ __forceinline__ int4 piece_at(const int4* __restrict__ recs, int32_t task, int32_t end,
                                         int G, int grp) {
  return task < end ? __ldg(recs + (int64_t)task * G + grp) : make_int4(0, 0, 0, 0);
}

// What a lane reads of a piece before it folds it: its part of the vertex's own
// row, as stored, and its ratings of the first two chunks.
template <int NR>
struct TaskHead {
  uint4 x[NR];
  uint32_t un, rn, um, rm;
  template <int K, int PREC, int LANES>
  __device__ __forceinline__ void load(const int4& rec, const void* __restrict__ self,
                                       const int32_t* __restrict__ nbr,
                                       const uint8_t* __restrict__ rate, const int (&dim)[NR],
                                       int sub) {
#pragma unroll
    for (int q = 0; q < NR; ++q) {
      x[q] = make_uint4(0u, 0u, 0u, 0u);
      if (rec.y > 0) x[q] = raw4<PREC>(self, (int64_t)rec.z * K + dim[q]);
    }
    un = rn = um = rm = 0u;
    if (sub < rec.y) {
      un = (uint32_t)__ldg(nbr + rec.x + sub);
      rn = __ldg(rate + rec.x + sub);
    }
    if (sub + LANES < rec.y) {
      um = (uint32_t)__ldg(nbr + rec.x + sub + LANES);
      rm = __ldg(rate + rec.x + sub + LANES);
    }
  }
};

template <int K, int PREC, bool SSE>
__global__ void __launch_bounds__(kCfSegThreads, 1)
cf_seg_kernel(RangeShare ranges, const int32_t* __restrict__ seg_task, int k, int32_t width,
              int32_t nn, const int4* __restrict__ recs, const int32_t* __restrict__ nbr,
              const uint8_t* __restrict__ rate, const void* __restrict__ self,
              const void* __restrict__ other, float* __restrict__ gpart,
              double* __restrict__ partials, unsigned* __restrict__ counter,
              double* __restrict__ sse_out) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int LANES = CfShape<K>::kLanes, NR = CfShape<K>::kReads, G = 32 / LANES;
  extern __shared__ __align__(16) float tab[];  // [width + 1][K], the last row zero
  __shared__ RangeSlots slots;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int sub = lane % LANES, grp = lane / LANES;
  int dim[NR];  // this lane's dimensions of a row: 4 from each
#pragma unroll
  for (int q = 0; q < NR; ++q)
    dim[q] = 4 * sub + (K / 2) * (LANES == 4 ? q ^ (grp & 1) : q);
  const char* tabq[NR];
#pragma unroll
  for (int q = 0; q < NR; ++q) tabq[q] = reinterpret_cast<const char*>(tab + dim[q]);
  for (int i = tid; i < K; i += kCfSegThreads) tab[width * K + i] = 0.0f;
  float se = 0.0f, sc = 0.0f;  // squared errors and what their FP32 sum has dropped
  int s = -1;
  int v = (int)blockIdx.x;
  int32_t t, hi, lo = 0;
  while (next_range(ranges, kCfSegThreads, &slots, &v, &t, &hi)) {
    while (t < hi) {
      const int sn = segment_of_task(seg_task, k, t);
      const int32_t te = __ldg(seg_task + sn + 1);
      if (sn != s) {
        s = sn;
        lo = s * width;
        const int nq = min(width, nn - lo) * (K / 4);
        __syncthreads();  // every warp is done with the previous table
#pragma unroll 4
        for (int i = tid; i < nq; i += kCfSegThreads)
          reinterpret_cast<float4*>(tab)[i] = load4<PREC>(other, (int64_t)lo * K + 4 * i);
        __syncthreads();
      }
      const int32_t e1 = min(hi, te);
      constexpr int kStep = kCfSegThreads / 32;
      // Three tasks are under way: this one is folded; the next one's vertex
      // rows and first ratings are on their way into registers; the places of
      // the one behind it are being read, so that these go into L2 early.
      int4 rec = piece_at(recs, t + w, e1, G, grp);
      int4 nrec = piece_at(recs, t + w + kStep, e1, G, grp);
      TaskHead<NR> cur, nxt;
      cur.load<K, PREC, LANES>(rec, self, nbr, rate, dim, sub);
      for (int32_t task = t + w; task < e1; task += kStep) {
        const int64_t slot = (int64_t)task * G + grp;
        const int len = rec.y;
        nxt.load<K, PREC, LANES>(nrec, self, nbr, rate, dim, sub);
        const int4 frec = piece_at(recs, task + 2 * kStep, e1, G, grp);
        u64 x[NR][2], g[NR][2];
#pragma unroll
        for (int q = 0; q < NR; ++q) {
          const float4 f = decode4<PREC>(cur.x[q]);
          x[q][0] = pair(f.x, f.y);
          x[q][1] = pair(f.z, f.w);
          g[q][0] = g[q][1] = 0ull;
        }
        const int chunks = (__shfl_sync(kFull, len, 0) + LANES - 1) / LANES;
        const int32_t* nb = nbr + rec.x + sub;
        const uint8_t* rt = rate + rec.x + sub;
        uint32_t un = cur.un, rn = cur.rn, um = cur.um, rm = cur.rm;
        float te2 = 0.0f;
        for (int c = 0; c < chunks; ++c) {
          const int i = c * LANES + sub;
          // row offset in the table, and the rating as FP32 (2^23 + r without its leading one)
          const uint32_t row = (i < len ? min(un - (uint32_t)lo, (uint32_t)width) : (uint32_t)width) * (4 * K);
          const float r = __uint_as_float(0x4B000000u | rn) - 8388608.0f;
          const bool real = i < len;
          un = um;
          rn = rm;
          if (i + 2 * LANES < len) {
            um = (uint32_t)__ldg(nb + (c + 2) * LANES);
            rm = __ldg(rt + (c + 2) * LANES);
          }
#pragma unroll
          for (int h = 0; h < LANES; h += 4) {  // four ratings of the group at a time
            ulonglong2 y[4][NR];
            float d[4];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const uint32_t at = __shfl_sync(kFull, row, (lane & ~(LANES - 1)) + h + j);
#pragma unroll
              for (int q = 0; q < NR; ++q)
                y[j][q] = *reinterpret_cast<const ulonglong2*>(tabq[q] + at);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              u64 a = mul2(x[0][0], y[j][0].x);
              fma2(a, x[0][1], y[j][0].y);
              fma2(a, x[1][0], y[j][1].x);
              fma2(a, x[1][1], y[j][1].y);
              d[j] = halves(a);
            }
            // the group's lanes add their parts and share the four ratings out:
            // lane sub ends up with the product of rating h + (sub & 3)
            const bool o1 = sub & 1, o2 = sub & 2;
            const float a01 = (o1 ? d[1] : d[0]) + __shfl_xor_sync(kFull, o1 ? d[0] : d[1], 1);
            const float a23 = (o1 ? d[3] : d[2]) + __shfl_xor_sync(kFull, o1 ? d[2] : d[3], 1);
            float dot = (o2 ? a23 : a01) + __shfl_xor_sync(kFull, o2 ? a01 : a23, 2);
            if (LANES == 8) dot += __shfl_xor_sync(kFull, dot, 4);
            float e;
            if (LANES == 4) {
              e = real ? r - dot : 0.0f;
              if (SSE) te2 = fmaf(e, e, te2);
            } else {  // lanes h .. h + 3 hold these ratings
              e = real ? r - dot : 0.0f;
              if (SSE && (sub & 4) == h) te2 = fmaf(e, e, te2);
            }
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float ej = __shfl_sync(kFull, e, (lane & ~(LANES - 1)) + h + j);
              const u64 e2 = pair(ej, ej);
#pragma unroll
              for (int q = 0; q < NR; ++q) {
                fma2(g[q][0], e2, y[j][q].x);
                fma2(g[q][1], e2, y[j][q].y);
              }
            }
          }
        }
        if (len > 0) {
#pragma unroll
          for (int q = 0; q < NR; ++q)
            __stcs(reinterpret_cast<ulonglong2*>(gpart + slot * K + dim[q]),
                   make_ulonglong2(g[q][0], g[q][1]));
        }
        if (frec.y > 0) {  // the pieces behind the next ones, into L2
          const char* at = reinterpret_cast<const char*>(nbr + frec.x);
          if (sub == 1) at = reinterpret_cast<const char*>(rate + frec.x);
          if (sub == 2)
            at = static_cast<const char*>(self) + (int64_t)frec.z * K * (PREC == 1 ? 2 : 4);
          if (sub == 3) at += min(4 * frec.y - 4, 128);
          asm volatile("prefetch.global.L2 [%0];" ::"l"(at));
        }
        rec = nrec;
        nrec = frec;
        cur = nxt;
        if (SSE) {  // compensated: the lane's sum runs over thousands of pieces
          const float a = se + te2, z = a - se;
          sc += (se - (a - z)) + (te2 - z);
          se = a;
        }
      }
      t = e1;
    }
  }
  if (!SSE) return;
  __shared__ double sh[32];
  __shared__ bool s_last;
  const double bs = block_sum<double, kCfSegThreads>((double)se + (double)sc, sh);
  if (tid == 0) {
    partials[blockIdx.x] = bs;
    __threadfence();
    s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double total = 0.0;
  for (int i = tid; i < (int)gridDim.x; i += kCfSegThreads) total += __ldcg(partials + i);
  total = block_sum<double, kCfSegThreads>(total, sh);
  if (tid == 0) {
    if (sse_out) *sse_out = total;
    *counter = 0u;
  }
}

// ---------------------------------------------------------------------------
// Building the pieces
// ---------------------------------------------------------------------------
constexpr int kWalkTile = 1024;  // ratings per warp

// Does a run begin at rating e (its vertex's first, or another segment than
// the rating before)?  Counts the runs of every warp's 1024 ratings, or (WRITE)
// lists their first ratings, vertices and segments.  *unsorted: a vertex whose
// segments do not ascend.
template <bool WRITE>
__global__ void __launch_bounds__(256)
cf_runs_kernel(const int64_t* __restrict__ off, int32_t n, int64_t R,
               const int32_t* __restrict__ nbr, uint32_t width, int32_t k,
               int32_t* __restrict__ cnt, const int64_t* __restrict__ first,
               int32_t* __restrict__ begin, int32_t* __restrict__ vtx, int32_t* __restrict__ seg,
               int32_t* __restrict__ unsorted) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5, nt = (R + kWalkTile - 1) / kWalkTile;
  RowWalk<int64_t> walk(off, n, (int32_t)R);
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nt; t += nw) {
    const int64_t b = t * kWalkTile;
    walk.seek((int32_t)b);
    int32_t before = b > 0 ? (int32_t)((uint32_t)__ldg(nbr + b - 1) / width) : -1;
    int64_t at = WRITE ? first[t] : 0;
    int c = 0;
    bool bad = false;
    for (int i = 0; i < kWalkTile && b + i < R; i += 32) {
      const int64_t e = b + i + lane;
      const bool ok = e < R;
      int32_t st, en;
      const int32_t r = walk.row_of((int32_t)e, ok, &st, &en);
      const int32_t s = ok ? (int32_t)((uint32_t)__ldcs(nbr + e) / width) : 0;
      int32_t p = __shfl_up_sync(0xffffffffu, s, 1);
      if (lane == 0) p = before;
      const bool head = ok && (st == (int32_t)e || s != p);
      bad = bad || (ok && (s >= k || (st != (int32_t)e && s < p)));
      const unsigned m = __ballot_sync(0xffffffffu, head);
      if (WRITE && head) {
        const int64_t j = at + __popc(m & ((1u << lane) - 1u));
        begin[j] = (int32_t)e;
        vtx[j] = r;
        seg[j] = s;
      }
      at += __popc(m);
      c += __popc(m);
      before = __shfl_sync(0xffffffffu, s, 31);
    }
    if (!WRITE) {
      if (lane == 0) cnt[t] = c;
      if (bad) atomicExch(unsorted, 1);
    }
  }
}

__global__ void cf_run_pieces_kernel(const int32_t* __restrict__ begin, int64_t nruns, int64_t R,
                                     int32_t* __restrict__ np) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nruns;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t end = i + 1 < nruns ? begin[i + 1] : R;
    np[i] = (int32_t)((end - begin[i] + kCfSegPiece - 1) / kCfSegPiece);
  }
}

// Sort keys of the runs' pieces and where each piece begins.
__global__ void cf_piece_kernel(const int32_t* __restrict__ begin, const int32_t* __restrict__ seg,
                                const int64_t* __restrict__ first, int64_t nruns, int64_t R,
                                uint32_t* __restrict__ key, int32_t* __restrict__ item,
                                int32_t* __restrict__ run) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nruns;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t end = i + 1 < nruns ? begin[i + 1] : R;
    const int64_t len = end - begin[i];
    for (int64_t p = first[i]; p < first[i + 1]; ++p) {
      const int64_t left = len - (p - first[i]) * kCfSegPiece;
      const int l = (int)(left < kCfSegPiece ? left : kCfSegPiece);
      key[p] = (uint32_t)seg[i] << kLenBits | (uint32_t)(kCfSegPiece - l);
      item[p] = (int32_t)p;
      run[p] = (int32_t)i;
    }
  }
}

// seg_item[s] = first sorted piece of segment s.
__global__ void cf_seg_start_kernel(const uint32_t* __restrict__ key, int64_t n, int k,
                                    int64_t* __restrict__ seg_item) {
  for (int s = blockIdx.x * blockDim.x + threadIdx.x; s <= k; s += gridDim.x * blockDim.x) {
    int64_t lo = 0, hi = n;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if ((int64_t)(key[mid] >> kLenBits) < s) lo = mid + 1; else hi = mid;
    }
    seg_item[s] = lo;
  }
}

// One thread per slot: its piece's record and the piece's slot.
__global__ void cf_slot_kernel(const int32_t* __restrict__ item, const int32_t* __restrict__ run,
                               const int64_t* __restrict__ run_first,
                               const int32_t* __restrict__ begin, const int32_t* __restrict__ vtx,
                               int64_t nruns, int64_t R, const int64_t* __restrict__ seg_item,
                               const int32_t* __restrict__ seg_task, int k, int G, int64_t nslots,
                               int4* __restrict__ recs, int32_t* __restrict__ slots) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nslots;
       q += (int64_t)gridDim.x * blockDim.x) {
    const int32_t t = (int32_t)(q / G);
    int lo = 0, hi = k + 1;  // last segment with seg_task <= t (empty ones share it)
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (seg_task[mid] <= t) lo = mid + 1; else hi = mid;
    }
    const int s = lo - 1;
    const int64_t i = seg_item[s] + (q - (int64_t)seg_task[s] * G);
    int4 rec = make_int4(0, 0, 0, 0);
    if (i < seg_item[s + 1]) {
      const int32_t p = item[i], r = run[p];
      const int64_t end = r + 1 < nruns ? begin[r + 1] : R;
      rec.x = begin[r] + (int32_t)(p - run_first[r]) * kCfSegPiece;
      rec.y = (int32_t)(end - rec.x < kCfSegPiece ? end - rec.x : kCfSegPiece);
      rec.z = vtx[r];
      slots[p] = (int32_t)q;
    }
    recs[q] = rec;
  }
}

// poff[v] = first piece of vertex v: that of its first run (runs lie in vertex
// order), found by the vertex's first rating.
__global__ void cf_poff_kernel(const int64_t* __restrict__ off, int64_t n,
                               const int32_t* __restrict__ begin, int64_t nruns,
                               const int64_t* __restrict__ run_first, int64_t* __restrict__ poff) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v <= n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t e = off[v];
    int64_t lo = 0, hi = nruns;
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (begin[mid] < e) lo = mid + 1; else hi = mid;
    }
    poff[v] = run_first[lo];
  }
}

// A task's cost: its longest piece and the fixed work around it.
__global__ void cf_cost_kernel(const int4* __restrict__ recs, int G, int32_t ntasks,
                               int32_t* __restrict__ cost) {
  for (int32_t t = blockIdx.x * blockDim.x + threadIdx.x; t < ntasks; t += gridDim.x * blockDim.x)
    cost[t] = recs[(int64_t)t * G].y + 8;
}

__global__ void cf_share_kernel(const int64_t* __restrict__ before, int32_t ntasks, int grid,
                                int32_t* __restrict__ blk_task) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b <= grid; b += gridDim.x * blockDim.x) {
    const int64_t want = before[ntasks] * b / grid;
    int32_t lo = 0, hi = ntasks;
    while (lo < hi) {
      const int32_t mid = (lo + hi) >> 1;
      if (before[mid] < want) lo = mid + 1; else hi = mid;
    }
    blk_task[b] = b == grid ? ntasks : lo;
  }
}

template <int K, int PREC>
int launch(const CfSegments& c, int64_t nn, const int32_t* nbr, const uint8_t* rate,
           const void* self, const void* other, float* gpart, bool with_sse, double* partials,
           unsigned* counter, double* sse, cudaStream_t s) {
  const size_t smem = sizeof(float) * K * ((size_t)c.width + 1);
  CG_CUDA(cudaMemsetAsync(c.next, 0, sizeof(unsigned) * c.grid, s));
  const RangeShare ranges{c.blk_task, c.next};
  if (with_sse) {
    auto fn = cf_seg_kernel<K, PREC, true>;
    CG_CUDA(cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    fn<<<c.grid, kCfSegThreads, smem, s>>>(ranges, c.seg_task, c.k, c.width, (int32_t)nn, c.recs,
                                           nbr, rate, self, other, gpart, partials, counter, sse);
  } else {
    auto fn = cf_seg_kernel<K, PREC, false>;
    CG_CUDA(cudaFuncSetAttribute((const void*)fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem));
    fn<<<c.grid, kCfSegThreads, smem, s>>>(ranges, c.seg_task, c.k, c.width, (int32_t)nn, c.recs,
                                           nbr, rate, self, other, gpart, nullptr, counter,
                                           nullptr);
  }
  CG_LAUNCH_CHECK();
  return CG_OK;
}

template <int K>
int launch_prec(const CfSegments& c, int precision, int64_t nn, const int32_t* nbr,
                const uint8_t* rate, const void* self, const void* other, float* gpart,
                bool with_sse, double* partials, unsigned* counter, double* sse, cudaStream_t s) {
  switch (precision) {
    case 0: return launch<K, 0>(c, nn, nbr, rate, self, other, gpart, with_sse, partials, counter, sse, s);
    case 1: return launch<K, 1>(c, nn, nbr, rate, self, other, gpart, with_sse, partials, counter, sse, s);
    default: return launch<K, 2>(c, nn, nbr, rate, self, other, gpart, with_sse, partials, counter, sse, s);
  }
}

}  // namespace

int cf_seg_gather(const CfSegments& c, int K, int precision, int64_t nn, const int32_t* nbr,
                  const uint8_t* rate, const void* self, const void* other, float* gpart,
                  bool with_sse, double* partials, unsigned* counter, double* sse,
                  cudaStream_t s) {
  switch (K) {
    case 32: return launch_prec<32>(c, precision, nn, nbr, rate, self, other, gpart, with_sse, partials, counter, sse, s);
    default: return launch_prec<64>(c, precision, nn, nbr, rate, self, other, gpart, with_sse, partials, counter, sse, s);
  }
}

int cf_seg_build(CfSegments* c, int64_t n, int64_t nn, int64_t R, int K, const int64_t* off,
                 const int32_t* nbr, cudaStream_t s) {
  *c = CfSegments();
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  // as many rows as fit next to the kernel's own shared memory and the zero row
  const int64_t cap = (int64_t)(di.smem_optin - 1024) / (4 * K) - 1;
  const int64_t k = ceil_div(nn, cap);
  if (K == 16 || R == 0 || R >= 0x7FFFFFFFLL - kWalkTile || n >= 0x7FFFFFFF || k > kCfSegMost) return CG_OK;
  const int32_t width = (int32_t)ceil_div(nn, k);
  const int G = pieces_per_task(K);
  const int64_t nt = ceil_div(R, kWalkTile);
  Scratch tmp(s, Scratch::round(4 * (size_t)nt) + Scratch::round(8 * (size_t)(nt + 1)) +
                     scan_scratch(nt) + 4096);
  int32_t *cnt = nullptr, *unsorted = nullptr;
  int64_t* first = nullptr;
  CG_CUDA(tmp.get(&cnt, nt));
  CG_CUDA(tmp.get(&first, nt + 1));
  CG_CUDA(tmp.get(&unsorted, 1));
  CG_CUDA(cudaMemsetAsync(unsorted, 0, sizeof(int32_t), s));
  const int wgrid = grid_for(nt * 32, 256);
  cf_runs_kernel<false><<<wgrid, 256, 0, s>>>(off, (int32_t)n, R, nbr, (uint32_t)width, (int32_t)k,
                                              cnt, nullptr, nullptr, nullptr, nullptr, unsorted);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i32_to_i64(cnt, first, nt, s, &tmp));
  int64_t nruns = 0;
  int32_t bad = 0;
  CG_CUDA(cudaMemcpyAsync(&nruns, first + nt, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaMemcpyAsync(&bad, unsorted, sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  // (ratings that are not grouped by segment would break into single ones)
  if (bad || !segments_pay(K, R, nruns, di.l2_bytes)) return CG_OK;
  const int64_t most = nruns + R / kCfSegPiece;  // pieces at most
  const size_t tasks = (size_t)(most / G + k);     // tasks at most
  Scratch t2(s, 4 * Scratch::round(4 * (size_t)nruns) + Scratch::round(8 * (size_t)(nruns + 1)) +
                    scan_scratch(nruns) + 5 * Scratch::round(4 * (size_t)most) +
                    sort_scratch(most) + Scratch::round(8 * (size_t)(k + 1)) +
                    Scratch::round(4 * tasks) + Scratch::round(8 * tasks + 8) +
                    scan_scratch((int64_t)tasks) + 8192);
  int32_t *begin = nullptr, *vtx = nullptr, *seg = nullptr, *np = nullptr, *item = nullptr,
          *sitem = nullptr, *run = nullptr;
  int64_t *run_first = nullptr, *seg_item = nullptr;
  uint32_t *key = nullptr, *skey = nullptr;
  CG_CUDA(t2.get(&begin, nruns));
  CG_CUDA(t2.get(&vtx, nruns));
  CG_CUDA(t2.get(&seg, nruns));
  CG_CUDA(t2.get(&np, nruns));
  CG_CUDA(t2.get(&run_first, nruns + 1));
  CG_CUDA(t2.get(&key, most));
  CG_CUDA(t2.get(&skey, most));
  CG_CUDA(t2.get(&item, most));
  CG_CUDA(t2.get(&sitem, most));
  CG_CUDA(t2.get(&run, most));
  CG_CUDA(t2.get(&seg_item, k + 1));
  cf_runs_kernel<true><<<wgrid, 256, 0, s>>>(off, (int32_t)n, R, nbr, (uint32_t)width, (int32_t)k,
                                             nullptr, first, begin, vtx, seg, nullptr);
  CG_LAUNCH_CHECK();
  cf_run_pieces_kernel<<<grid_for(nruns, 256), 256, 0, s>>>(begin, nruns, R, np);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i32_to_i64(np, run_first, nruns, s, &t2));
  cf_piece_kernel<<<grid_for(nruns, 256), 256, 0, s>>>(begin, seg, run_first, nruns, R, key, item,
                                                       run);
  CG_LAUNCH_CHECK();
  int64_t npieces = 0;
  CG_CUDA(cudaMemcpyAsync(&npieces, run_first + nruns, sizeof(int64_t), cudaMemcpyDeviceToHost,
                          s));
  CG_CUDA(cudaStreamSynchronize(s));
  int bits = kLenBits;
  while (((int64_t)1 << bits) < k << kLenBits) ++bits;
  CG_TRY(radix_sort_pairs(key, item, skey, sitem, npieces, bits, s, &t2));
  cf_seg_start_kernel<<<grid_for(k + 1, 128), 128, 0, s>>>(skey, npieces, (int)k, seg_item);
  CG_LAUNCH_CHECK();
  std::vector<int64_t> hs(k + 1);
  CG_CUDA(cudaMemcpyAsync(hs.data(), seg_item, sizeof(int64_t) * (k + 1), cudaMemcpyDeviceToHost,
                          s));
  CG_CUDA(cudaStreamSynchronize(s));
  std::vector<int32_t> task(k + 1, 0);
  for (int64_t q = 0; q < k; ++q) task[q + 1] = task[q] + (int32_t)ceil_div(hs[q + 1] - hs[q], G);
  c->ntasks = task[k];
  c->npieces = npieces;
  c->nslots = (int64_t)c->ntasks * G;
  c->grid = std::max(1, std::min(c->ntasks, di.sm_count));
  const size_t rb = Scratch::round(16 * (size_t)c->nslots), sb = Scratch::round(4 * (size_t)npieces),
               pb = Scratch::round(8 * (size_t)(n + 1)), tb = Scratch::round(4 * (size_t)(k + 1)),
               gb = Scratch::round(4 * (size_t)(c->grid + 1));
  c->bytes = (int64_t)(rb + sb + pb + tb + 2 * gb);
  CG_CUDA(cudaMalloc((void**)&c->slab, (size_t)c->bytes));
  c->recs = reinterpret_cast<int4*>(c->slab);
  c->slots = reinterpret_cast<int32_t*>(c->slab + rb);
  c->poff = reinterpret_cast<int64_t*>(c->slab + rb + sb);
  c->seg_task = reinterpret_cast<int32_t*>(c->slab + rb + sb + pb);
  c->blk_task = reinterpret_cast<int32_t*>(c->slab + rb + sb + pb + tb);
  c->next = reinterpret_cast<unsigned*>(c->slab + rb + sb + pb + tb + gb);
  CG_CUDA(cudaMemcpyAsync(c->seg_task, task.data(), sizeof(int32_t) * (k + 1),
                          cudaMemcpyHostToDevice, s));
  cf_slot_kernel<<<grid_for(c->nslots, 256), 256, 0, s>>>(
      sitem, run, run_first, begin, vtx, nruns, R, seg_item, c->seg_task, (int)k, G, c->nslots,
      c->recs, c->slots);
  CG_LAUNCH_CHECK();
  cf_poff_kernel<<<grid_for(n + 1, 256), 256, 0, s>>>(off, n, begin, nruns, run_first, c->poff);
  CG_LAUNCH_CHECK();
  int32_t* cost = nullptr;
  int64_t* before = nullptr;
  CG_CUDA(t2.get(&cost, c->ntasks));
  CG_CUDA(t2.get(&before, (size_t)c->ntasks + 1));
  cf_cost_kernel<<<grid_for(c->ntasks, 256), 256, 0, s>>>(c->recs, G, c->ntasks, cost);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i32_to_i64(cost, before, c->ntasks, s, &t2));
  cf_share_kernel<<<grid_for(c->grid + 1, 128), 128, 0, s>>>(before, c->ntasks, c->grid,
                                                              c->blk_task);
  CG_LAUNCH_CHECK();
  CG_CUDA(cudaStreamSynchronize(s));
  c->width = width;
  c->k = (int32_t)k;
  return CG_OK;
}

void cf_seg_free(CfSegments* c) {
  cudaFree(c->slab);
  *c = CfSegments();
}

}  // namespace cg
