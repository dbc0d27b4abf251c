// The edge stream of the staged segments (their source values sit in a
// shared-memory table) and the warp code that folds it.
//
// What bounded the earlier layout (512 consecutive edges per warp chunk, a
// row-end mask per lane, a segmented scan per chunk): instructions and the
// dependent chain of every chunk.  Each of a lane's 16 edges cost a test of
// its row-end bit and a divergent row store, about 25 instructions per edge
// slot, while the shared-memory lookups themselves take one.
//
// Here rows are grouped by length.  The rows of a window (kStagedWindow
// consecutive subgraph rows of one segment) are sorted by a length class,
// and a warp task holds rows of one class only, so its shape is known before
// its edges are read: no flags, no scan, no divergence.
//   classes 0..7    rows of exactly L = class + 1 edges; a lane folds R of
//                   them (R L <= 16 edges per lane);
//   classes 8..15   rows of 9..16 edges, one per lane;
//   classes 16..55  rows of 17..512 edges on g = 2..32 adjacent lanes, t = 9..16
//                   edges per lane (an eighth at most is padding), then log2(g)
//                   shuffles;
//   classes 56..69  rows of 513..4096 edges on the whole warp, t = 24, 32, ..128;
//   class 70        4096 edges of a longer row: the sum goes to a carry slot and
//                   the fix-up adds it to the row (the row's remaining 1..4096
//                   edges are an ordinary row of their class).
// A task's indices are 16-bit, two slots per 32-bit word, four words of a lane
// together (16-byte loads) and the lanes adjacent, padded with the index of a
// table entry that holds the operator's identity.  Behind them lie the rows'
// 16-bit positions in the window: the sums go to their rows' canonical
// places.  Short rows are so frequent that a store still fills its sectors
// (RMAT-22: 0.47 sectors per row), and 32,768 rows per window keep the
// partly filled tasks at 3% of the slots.
//
// Measured (one staged launch; the earlier layout and schedule, then this):
// 528.7 M edges 562 -> 394 us, 65.2 M edges 89 -> 63 us, 15.7 M edges 26.7 ->
// 26.9 us (one table: its copy and the launch are a third of that).  On 130 M
// edges 84 M -> 42 M instructions (ncu); what is left is bound by the shared-memory
// pipe (3.9 wavefronts per random lookup, 64% of its peak over the launch of 264 M
// edges in 19 segments) and by the latency of a task's stream loads.  Loading the next task's words into registers first
// cost more instructions than it hid (423 us), the prefetch distance is flat
// from 32 to 160 KB and worth 10% of the launch against none.
#pragma once

#include "seg_gather.cuh"

namespace cg {

constexpr int kStagedWindow = 32768;  // rows per sorting window (16-bit positions)
constexpr int kStagedMost = 4096;     // edges of a row one task folds
constexpr int kClassBits = 7;
constexpr int kClassFull = 70;        // a full piece of a longer row
constexpr int kStreamAhead = 64 * 1024;  // the stream is pulled into L2 this many bytes ahead
constexpr uint32_t kNoRow = 0xFFFFu;  // position of an unused row slot

// rows folded by one lane of classes 0..7 (R * (class + 1) <= 16)
__host__ __device__ constexpr int short_rows(int c) {
  return c == 0 ? 8 : c == 1 ? 8 : c == 2 ? 5 : c == 3 ? 4 : c == 4 ? 3 : 2;
}

// Length class of a row of len edges, 1 <= len <= kStagedMost.
__host__ __device__ inline int staged_class(int len) {
  if (len <= 16) return len - 1;
  if (len <= 512) {
    int j = 1;
    while (len > (16 << j)) ++j;
    return 16 + (j - 1) * 8 + ((len + (1 << j) - 1) >> j) - 9;
  }
  return 56 + (len + 255) / 256 - 3;
}

// log2 of the lanes that share a row
__host__ __device__ inline int class_lg(int c) { return c < 16 ? 0 : c < 56 ? (c - 16) / 8 + 1 : 5; }
// edge slots per lane
__host__ __device__ inline int class_slots(int c) {
  return c < 8 ? short_rows(c) * (c + 1)
               : c < 16 ? c + 1 : c < 56 ? 9 + (c - 16) % 8 : c < kClassFull ? 24 + 8 * (c - 56) : 128;
}
// 32-bit words per lane: 4, 6 or 8 (4 lie together, then 2 or 4), or a multiple of 4
__host__ __device__ inline int class_words(int c) {
  const int w = (class_slots(c) + 1) >> 1;
  return w + (w & 1);
}
// words of row positions per lane (0: 16 bits per row)
__host__ __device__ inline int class_pos(int c) { return c < 3 ? 4 : c < 5 ? 2 : c < 8 ? 1 : 0; }
// rows of a task
__host__ __device__ inline int class_rows(int c) {
  return c < 8 ? 32 * short_rows(c) : 32 >> class_lg(c);
}
// 32-byte units of a task: its index words, then its rows' positions
__host__ __device__ inline int class_units(int c) {
  return 4 * class_words(c) + (c < 8 ? 4 * class_pos(c) : c < 16 ? 2 : 1);
}
// Where word i of lane `lane` lies in a task (in words).
__host__ __device__ inline int word_at(int words, int i, int lane) {
  const int q = i & ~3;                       // groups of four words, 16 bytes per lane
  const int n = words - q >= 4 ? 4 : words - q;  // the last group may hold two
  return q * 32 + lane * n + (i & 3);
}
// the code path of a class: 0..7 short rows, 8..11 rows on 1..32 lanes with
// 9-10, 11-12, 13-14, 15-16 slots, then one long row and a full piece
constexpr uint32_t kShapeLong = 12, kShapeFull = 13;
__host__ __device__ inline uint32_t class_shape(int c) {
  return c < 8 ? c : c < 56 ? 3 + (class_slots(c) + 1) / 2 : c < kClassFull ? kShapeLong : kShapeFull;
}
// A task's descriptor word: shape | log2 lanes << 4 | words << 8 | units << 16.
__host__ __device__ inline uint32_t class_word(int c) {
  return class_shape(c) | (uint32_t)class_lg(c) << 4 | (uint32_t)class_words(c) << 8 |
         (uint32_t)class_units(c) << 16;
}

#ifdef __CUDACC__

// The tasks of the staged launches.  A descriptor: (stream offset in 32-byte
// units, class_word, first row of the window (the carry slot of a full
// piece), -).
struct StagedTasks {
  const uint8_t* cs;        // the stream
  const uint4* desc;        // one descriptor per task
  const int32_t* seg_task;  // [k+1] first task of each segment
  int32_t pad;              // table entry that holds the identity
};

// A lane's first 8 words of a task (fewer where the task has fewer).
__device__ __forceinline__ void load_words(const uint8_t* base, uint32_t word,
                                           uint32_t (&w)[8]) {
  const int lane = threadIdx.x & 31;
  const int nw = (int)((word >> 8) & 0xFFu);
  const uint4 a = __ldcs(reinterpret_cast<const uint4*>(base) + lane);
  w[0] = a.x; w[1] = a.y; w[2] = a.z; w[3] = a.w;
  if (nw >= 8) {
    const uint4 b = __ldcs(reinterpret_cast<const uint4*>(base + 512) + lane);
    w[4] = b.x; w[5] = b.y; w[6] = b.z; w[7] = b.w;
  } else if (nw == 6) {
    const uint2 b = __ldcs(reinterpret_cast<const uint2*>(base + 512) + lane);
    w[4] = b.x; w[5] = b.y;
  }
}

// A lane's R rows of L edges each; pp: the rows' positions.
template <class Op, int L>
__device__ __forceinline__ void short_rows_task(const uint32_t (&w)[8],
                                                const uint8_t* pp,
                                                const typename Op::T* tab,
                                                typename Op::T* __restrict__ out) {
  using T = typename Op::T;
  constexpr int R = short_rows(L - 1), NP = L <= 3 ? 4 : L <= 5 ? 2 : 1;
  const int lane = threadIdx.x & 31;
  uint32_t pos[4];
  if constexpr (NP == 4) {
    const uint4 b = __ldcs(reinterpret_cast<const uint4*>(pp) + lane);
    pos[0] = b.x; pos[1] = b.y; pos[2] = b.z; pos[3] = b.w;
  } else if constexpr (NP == 2) {
    const uint2 b = __ldcs(reinterpret_cast<const uint2*>(pp) + lane);
    pos[0] = b.x; pos[1] = b.y;
  } else {
    pos[0] = __ldcs(reinterpret_cast<const unsigned*>(pp) + lane);
  }
  T a[R];
#pragma unroll
  for (int q = 0; q < R; ++q) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const int e = q * L + l;
      const T v = tab[(e & 1) ? w[e >> 1] >> 16 : w[e >> 1] & 0xFFFFu];
      a[q] = l == 0 ? v : Op::op(a[q], v);
    }
  }
#pragma unroll
  for (int q = 0; q < R; ++q) {
    const uint32_t id = (q & 1) ? pos[q >> 1] >> 16 : pos[q >> 1] & 0xFFFFu;
    if (id != kNoRow) out[id] = a[q];
  }
}

// Adds both halves of words [0, NW) to a and b.
template <class Op, int NW>
__device__ __forceinline__ void fold_words(const uint32_t (&w)[8], const typename Op::T* tab,
                                           typename Op::T& a, typename Op::T& b) {
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    a = Op::op(a, tab[w[i] & 0xFFFFu]);
    b = Op::op(b, tab[w[i] >> 16]);
  }
}

// Rows on 2^lg adjacent lanes each, NW words per lane; pp: their positions.
template <class Op, int NW>
__device__ __forceinline__ void lane_rows_task(const uint32_t (&w)[8],
                                               const uint8_t* pp, int lg,
                                               const typename Op::T* tab,
                                               typename Op::T* __restrict__ out) {
  using T = typename Op::T;
  const int lane = threadIdx.x & 31;
  const uint32_t id = __ldcs(reinterpret_cast<const unsigned short*>(pp) + (lane >> lg));
  T a = Op::identity(), b = Op::identity();
  fold_words<Op, NW>(w, tab, a, b);
  T v = Op::op(a, b);
  for (int o = 1; o < (1 << lg); o <<= 1) v = Op::op(v, __shfl_xor_sync(0xffffffffu, v, o));
  if ((lane & ((1 << lg) - 1)) == 0 && id != kNoRow) out[id] = v;
}

// One task (at base) whose first words are loaded.
template <class Op>
__device__ __forceinline__ void fold_task(const uint8_t* base, uint32_t word,
                                          int32_t row, const uint32_t (&w)[8],
                                          const typename Op::T* tab,
                                          typename Op::T* __restrict__ out,
                                          typename Op::T* __restrict__ carry) {
  using T = typename Op::T;
  T* rows = out + row;
  const int lg = (word >> 4) & 15;
  const int nw = (int)((word >> 8) & 0xFFu);
  const uint8_t* pp = base + nw * 128;
  switch (word & 15u) {  // uniform in the warp
    case 0: short_rows_task<Op, 1>(w, pp, tab, rows); return;
    case 1: short_rows_task<Op, 2>(w, pp, tab, rows); return;
    case 2: short_rows_task<Op, 3>(w, pp, tab, rows); return;
    case 3: short_rows_task<Op, 4>(w, pp, tab, rows); return;
    case 4: short_rows_task<Op, 5>(w, pp, tab, rows); return;
    case 5: short_rows_task<Op, 6>(w, pp, tab, rows); return;
    case 6: short_rows_task<Op, 7>(w, pp, tab, rows); return;
    case 7: short_rows_task<Op, 8>(w, pp, tab, rows); return;
    case 8: lane_rows_task<Op, 5>(w, pp, lg, tab, rows); return;
    case 9: lane_rows_task<Op, 6>(w, pp, lg, tab, rows); return;
    case 10: lane_rows_task<Op, 7>(w, pp, lg, tab, rows); return;
    case 11: lane_rows_task<Op, 8>(w, pp, lg, tab, rows); return;
    default: break;
  }
  // one long row (or a full piece of one) on the whole warp: 12 words and more
  const int lane = threadIdx.x & 31;
  T a = Op::identity(), b = Op::identity();
  fold_words<Op, 8>(w, tab, a, b);
  const uint4* p = reinterpret_cast<const uint4*>(base) + lane;
  for (int i = 8; i < nw; i += 8) {
    uint32_t u[8];
    const uint4 x = __ldcs(p + i * 8);
    u[0] = x.x; u[1] = x.y; u[2] = x.z; u[3] = x.w;
    if (i + 4 < nw) {
      const uint4 y = __ldcs(p + (i + 4) * 8);
      u[4] = y.x; u[5] = y.y; u[6] = y.z; u[7] = y.w;
      fold_words<Op, 8>(u, tab, a, b);
    } else {
      fold_words<Op, 4>(u, tab, a, b);
    }
  }
  T v = Op::op(a, b);
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) v = Op::op(v, __shfl_xor_sync(0xffffffffu, v, o));
  if (lane == 0) {
    if ((word & 15u) == kShapeFull)
      carry[row] = v;
    else
      rows[__ldcs(reinterpret_cast<const unsigned short*>(pp))] = v;
  }
}

// Bulk prefetch of [p, p + bytes) into L2 (TMA; p and bytes 16-byte aligned).
__device__ __forceinline__ void prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Tasks [t0, t1) by a block's warps [0, warps), round robin; each reads its
// task's descriptor one turn ahead.  Warp 0 has the stream kStreamAhead bytes
// behind the tasks of its turn pulled into L2 (the tasks tile the stream, so
// the shifted stretches tile it too; the stream is allocated with that much
// room behind it).
template <class Op>
__device__ __forceinline__ void staged_run(const StagedTasks& q, int32_t t0, int32_t t1,
                                           int w, int warps, const typename Op::T* tab,
                                           typename Op::T* __restrict__ out,
                                           typename Op::T* __restrict__ carry) {
  int32_t t = t0 + w;
  if (t >= t1) return;
  uint4 d = __ldca(q.desc + t);
  for (;;) {
    const uint8_t* base = q.cs + (size_t)d.x * 32;
    uint32_t c[8];
    load_words(base, d.y, c);
    const int32_t tn = t + warps;
    const uint4 dn = __ldca(q.desc + min(tn, t1 - 1));
    if (threadIdx.x == 0 && dn.x > d.x)
      prefetch_l2(base + kStreamAhead, min((dn.x - d.x) * 32, (uint32_t)kStreamAhead));
    fold_task<Op>(base, d.y, (int32_t)d.z, c, tab, out, carry);
    if (tn >= t1) break;
    t = tn;
    d = dn;
  }
}

#endif  // __CUDACC__

}  // namespace cg
