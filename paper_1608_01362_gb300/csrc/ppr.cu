// Batched personalised PageRank: 64 rank vectors advanced together over one
// segmented graph.  Each iteration is Algorithm 3's gather and Algorithm 4's
// merge with 64-wide rows in place of scalars (an SpMM with a 64-column dense
// operand), followed by the personalised form of Algorithm 5's update:
//   R'[v][j] = d (sum_{u->v} C[u][j]) + [v == seed_j] ((1-d) + d D_j)
//   C'[v][j] = R'[v][j] / outdeg(v),     D'_j = sum_{outdeg(v)=0} R'[v][j]
// (the teleport and the dangling mass of column j return to its seed).
//
// Storage.  The iteration state is C (the contributions R/outdeg) of the
// non-dangling vertices: with two planes FP32, 256 bytes per vertex (the bytes
// of a BF16 hi + lo pair, at full precision: an edge is then four packed adds
// and no unpacking), with one plane BF16, 128 bytes.  Gathers accumulate in
// FP32.  R itself is written in FP32 only when asked for (the last iteration,
// and the one before it for the L1 residual); D_j and the residual are FP64
// with a fixed reduction order.
//
// Kernels per iteration:
//   ppr_gather_kernel  an octet (8 lanes, 8 columns each) walks a 128-edge
//                      chunk of one segment's flagged edge stream, reading
//                      C rows of the segment's sources (a slice sized to
//                      stay in L2), and writes each subgraph row's 64 sums
//                      to intermBuf; the row open at the chunk's end goes
//                      to a carry slot;
//   ppr_fixup_kernel   completes the rows that span chunks: each run of
//                      carries (consecutive chunks open on the same row, a
//                      static structure) is cut into pieces of <= 16 chunks
//                      summed in parallel; the last piece of a run adds the
//                      pieces' sums, in order, into the row;
//   ppr_merge_kernel   an octet takes 16 consecutive destinations, sums
//                      their intermBuf rows (destination-major list of the
//                      rows, in segment order), applies the update and
//                      writes C' (and R'), with per-column FP64 partials
//                      reduced by the last block.
#include "ppr.cuh"

namespace cg {
namespace {

// BF16 pairs (element 0 in the low half) to FP32: exact.
__device__ __forceinline__ float bf_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float bf_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// 8 FP32 values as 4 packed pairs: one 32-byte load, four packed adds
// (rounded as the scalar ones).
struct Row8 {
  uint64_t p[4];
};

__device__ __forceinline__ uint64_t pair(float a, float b) {
  return (uint64_t)__float_as_uint(b) << 32 | __float_as_uint(a);
}

__device__ __forceinline__ void add_row(Row8& acc, const Row8& x) {
#pragma unroll
  for (int q = 0; q < 4; ++q)
    asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc.p[q]) : "l"(x.p[q]));
}

// Columns 8 lane8 .. 8 lane8 + 7 of a contribution row.  FP32 rows are not kept
// in L1: hardly one in eight is read again in time (274 us against 261 for a
// gather of 15.7 M edges), and the edge words want the room.
template <int PLANES>
__device__ __forceinline__ Row8 load_contrib(const void* c, uint32_t row, int lane8) {
  Row8 x;
  if (PLANES == 2) {
    const float* p = static_cast<const float*>(c) + ((int64_t)row * kCols + lane8 * 8);
    asm volatile("ld.global.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];"
                 : "=l"(x.p[0]), "=l"(x.p[1]), "=l"(x.p[2]), "=l"(x.p[3])
                 : "l"(p));
  } else {
    const uint4 h = __ldca(static_cast<const uint4*>(c) + ((int64_t)row * 8 + lane8));
    x.p[0] = pair(bf_lo(h.x), bf_hi(h.x));
    x.p[1] = pair(bf_lo(h.y), bf_hi(h.y));
    x.p[2] = pair(bf_lo(h.z), bf_hi(h.z));
    x.p[3] = pair(bf_lo(h.w), bf_hi(h.w));
  }
  return x;
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// An octet's row moves in 32-byte pieces, one instruction and whole sectors a
// lane; streaming (evict-first): intermBuf and carries must not push the
// segment's C rows out of L2.
__device__ __forceinline__ void store_row(float* dst, const Row8& a) {
  asm volatile("st.global.cs.v4.b64 [%0], {%1, %2, %3, %4};" ::"l"(dst), "l"(a.p[0]), "l"(a.p[1]),
               "l"(a.p[2]), "l"(a.p[3])
               : "memory");
}

__device__ __forceinline__ Row8 load_row(const float* src) {
  Row8 x;
  asm volatile("ld.global.cs.v4.b64 {%0, %1, %2, %3}, [%4];"
               : "=l"(x.p[0]), "=l"(x.p[1]), "=l"(x.p[2]), "=l"(x.p[3])
               : "l"(src)
               : "memory");
  return x;
}

__device__ __forceinline__ void unpack(const Row8& a, float (&x)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = __uint_as_float((uint32_t)(a.p[q >> 1] >> (32 * (q & 1))));
}

__device__ __forceinline__ Row8 pack(const float (&x)[8]) {
  return {{pair(x[0], x[1]), pair(x[2], x[3]), pair(x[4], x[5]), pair(x[6], x[7])}};
}

template <int PLANES>
__device__ __forceinline__ void store_contrib(void* c, int64_t v, int lane8, const float (&x)[8]) {
  if (PLANES == 2)
    store_row(static_cast<float*>(c) + v * kCols + lane8 * 8, pack(x));
  else
    __stcs(static_cast<uint4*>(c) + v * 8 + lane8,
           make_uint4(pack_bf16(x[0], x[1]), pack_bf16(x[2], x[3]), pack_bf16(x[4], x[5]),
                      pack_bf16(x[6], x[7])));
}

// ---------------------------------------------------------------------------
// Gather (Algorithm 3, 64-wide).  Octet o takes chunks o, o + #octets, ...:
// all octets sweep the chunks in segment order together, so the C rows read
// at any moment belong to one or two segments' source slices.
//
// What bounds it is the row reads' way from L2: 256 bytes an edge at 64 bytes
// per cycle and SM, 215 us for 15.7 M edges at 1.92 GHz (two planes); the
// kernel takes 246.  Reading rows as two BF16 planes it took 335: 67
// instructions for four octets' edge, 32 of them unpacking.  Rows in flight
// per octet beyond the one or two that fit in 40 registers, or more than 6
// blocks per SM, cost (two rows at 5 blocks 316 us, 7 blocks 296): they evict
// one another from L2 and the edge words from L1.  One plane's rows are half as
// long and take 8 blocks (uniform graph of 1 M vertices and 16 M edges in 4 segments
// 446 us, 477 with 6; RMAT of as many 227 and 226; 4 M uniform edges 129 and 198).
// ---------------------------------------------------------------------------
template <int PLANES>
__global__ void __launch_bounds__(kThreads, kGatherBlocks[PLANES])
ppr_gather_kernel(const uint32_t* colf, const PprSeg* segs,
                  const int2* chunks, int64_t nchunks, const void* contrib,
                  float* interm, float* carry) {
  if (!chain_begin()) return;
  const int lane8 = threadIdx.x & 7;
  const int noct = (int)((gridDim.x * blockDim.x) >> 3);
  for (int c = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 3); c < (int)nchunks; c += noct) {
    const int2 ch = __ldca(chunks + c);
    const PprSeg sg = segs[ch.y];
    const int64_t el = (c - sg.chunk0) * kChunk;
    const int n = (int)min((int64_t)kChunk, (int64_t)sg.E - el);
    const uint4* cf = reinterpret_cast<const uint4*>(colf + sg.cstart + el);
    int32_t row = ch.x;
    Row8 acc = {{0, 0, 0, 0}};
    for (int g = 0; g < n; g += 4, ++cf) {
      const uint4 f4 = __ldca(cf);  // the octet's lanes read the same four edges
      const uint32_t f[4] = {f4.x, f4.y, f4.z, f4.w};
      if (g + 4 <= n && !((f4.x | f4.y | f4.z | f4.w) & kRowEnd)) {
#pragma unroll
        for (int u = 0; u < 4; ++u)
          add_row(acc, load_contrib<PLANES>(contrib, sg.lo + f[u], lane8));
        continue;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if (g + u < n) {
          add_row(acc, load_contrib<PLANES>(contrib, sg.lo + (f[u] & ~kRowEnd), lane8));
          if (f[u] & kRowEnd) {
            store_row(interm + (int64_t)row * kCols + lane8 * 8, acc);
            ++row;
            acc = {{0, 0, 0, 0}};
          }
        }
      }
    }
    // the row open at the chunk's end
    if (!(__ldca(colf + sg.cstart + el + n - 1) & kRowEnd))
      store_row(carry + (int64_t)c * kCols + lane8 * 8, acc);
  }
}

// The sum of n rows, in order, four of them in flight (they are read past L1:
// another octet may have written them in this launch).
__device__ __forceinline__ void sum_rows(const float* src, int n, float (&sum)[8]) {
  constexpr int U = 4;
#pragma unroll
  for (int q = 0; q < 8; ++q) sum[q] = 0.0f;
  for (int j = 0; j < n; j += U) {
    float4 a[U], b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = b[u] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (j + u < n) {
        const float4* p = reinterpret_cast<const float4*>(src + (int64_t)(j + u) * kCols);
        a[u] = __ldcg(p);
        b[u] = __ldcg(p + 1);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      if (j + u >= n) break;
      sum[0] += a[u].x; sum[1] += a[u].y; sum[2] += a[u].z; sum[3] += a[u].w;
      sum[4] += b[u].x; sum[5] += b[u].y; sum[6] += b[u].z; sum[7] += b[u].w;
    }
  }
}

// Rows that span chunks.  One octet per piece (<= kPprPiece consecutive chunks
// of one run): it sums the chunks' carries in order.  A run of one piece adds
// its sum into the row directly; otherwise each piece stores its sum and the
// last piece of the run to finish (atomic count, no waiting) adds the pieces'
// sums in piece order into the row -- deterministic, and a hub row spanning
// thousands of chunks does not hold up one octet.  What bounds it is that
// chain of reads, so pieces are short and their rows read four at a time (23.8
// us with pieces of 32 read one by one, 10.1 so, at 122,657 chunks).
__global__ void __launch_bounds__(kThreads)
ppr_fixup_kernel(const int4* pieces, int64_t npieces, const int4* runs,
                 const float* carry, float* piece_sum,
                 unsigned* run_done, float* interm) {
  if (!chain_begin()) return;
  const int lane8 = threadIdx.x & 7;
  const unsigned omask = 0xffu << (threadIdx.x & 24);
  const int64_t noct = ((int64_t)gridDim.x * blockDim.x) >> 3;
  for (int64_t p = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 3; p < npieces;
       p += noct) {
    const int4 pc = __ldca(pieces + p);  // (first chunk, chunks, run)
    const int4 rn = __ldca(runs + pc.z); // (row, first piece, pieces)
    float sum[8], x[8];
    sum_rows(carry + (int64_t)pc.x * kCols + lane8 * 8, pc.y, sum);
    float* dst = interm + (int64_t)rn.x * kCols + lane8 * 8;
    if (rn.z == 1) {
      unpack(load_row(dst), x);
#pragma unroll
      for (int q = 0; q < 8; ++q) x[q] += sum[q];
      store_row(dst, pack(x));
      continue;
    }
    store_row(piece_sum + p * kCols + lane8 * 8, pack(sum));
    __threadfence();
    __syncwarp(omask);
    unsigned prev = 0;
    if (lane8 == 0) prev = atomicAdd(run_done + pc.z, 1u);
    prev = __shfl_sync(omask, prev, 0, 8);
    if (prev != (unsigned)rn.z - 1) continue;  // not the run's last piece
    __threadfence();
    float tot[8];
    sum_rows(piece_sum + (int64_t)rn.y * kCols + lane8 * 8, rn.z, tot);
    unpack(load_row(dst), x);
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] += tot[q];
    store_row(dst, pack(x));
    if (lane8 == 0) run_done[pc.z] = 0u;  // ready for the next iteration
  }
}

// ---------------------------------------------------------------------------
// Merge (Algorithm 4, destination-major) fused with the personalised update.
//
// What bounds it is memory: its rows once in, the contributions once out (38 us
// of the 69 it takes at 1 M vertices and 15.7 M edges), and the reads in flight
// towards that: the first rows of an octet's next two destinations, 24 warps
// per SM (with 32 and spills 71 us, with one row ahead 75).  The octets of a
// warp go through their destinations together, so the update runs once for
// four.  FP64 sums lie in shared memory, touched only where there is something
// to add.
// ---------------------------------------------------------------------------
struct MergeArgs {
  const int32_t* dst_off;
  const int32_t* dst_rows;
  const float* interm;
  const float* inv;
  const int32_t* seeds;
  const uint32_t* seed_bits;
  void* contrib;
  float* r_out;        // NULL: R' not written
  const float* r_old;  // NULL: no residual
  double* D;           // [64] in: D of the previous iterate; out: D'
  double* resid;       // [64] or NULL
  double* partials;    // [grid][128], then the groups' sums [ceil(grid / 32)][128]
  unsigned* counter;   // groups finished, then each group's finished blocks
  float d;
  int32_t V;
};

template <int PLANES, bool RESID>
__global__ void __launch_bounds__(kThreads, 3)
ppr_merge_kernel(MergeArgs a) {
  __shared__ float s_tele[kCols];
  __shared__ int32_t s_seed[kCols];
  // per warp and lane: the FP64 sums of its columns 8 lane8 + q
  __shared__ double s_acc[kThreads / 32][RESID ? 2 : 1][8][32];
  __shared__ double s_half[2 * kCols];
  __shared__ bool s_last;
  if (!chain_begin()) return;
  if (threadIdx.x < kCols) {
    s_tele[threadIdx.x] =
        (float)((1.0 - (double)a.d) + (double)a.d * a.D[threadIdx.x]);
    s_seed[threadIdx.x] = a.seeds[threadIdx.x];
  }
  __syncthreads();
  const int lane8 = threadIdx.x & 7;
  const int64_t noct = ((int64_t)gridDim.x * blockDim.x) >> 3;
  const int oct = (threadIdx.x >> 3) & 3;
  const int64_t ntask = ((int64_t)a.V + kTask - 1) / kTask;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    s_acc[w][0][q][lane] = 0.0;
    if (RESID) s_acc[w][RESID][q][lane] = 0.0;
  }
  for (int64_t t0 = (((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5) * 4; t0 < ntask;
       t0 += noct) {
    // (an octet past the last task has no destinations)
    const int64_t v0 = min((t0 + oct) * kTask, (int64_t)a.V);
    const int nv = (int)min((int64_t)kTask, (int64_t)a.V - v0);
    // row-list offsets, first rows and reciprocal degrees of the destinations
    const int32_t off_a = __ldca(a.dst_off + v0 + min(lane8, nv));
    const int32_t off_b = __ldca(a.dst_off + v0 + min(8 + lane8, nv));
    const float inv_a = lane8 < nv ? __ldca(a.inv + v0 + lane8) : 0.0f;
    const float inv_b = 8 + lane8 < nv ? __ldca(a.inv + v0 + 8 + lane8) : 0.0f;
    const uint32_t sbits = nv > 0 ? __ldca(a.seed_bits + (v0 >> 5)) >> (v0 & 31) : 0u;
    const int32_t o_end = __ldca(a.dst_off + v0 + nv);
    const int32_t row_a = off_a < o_end ? __ldca(a.dst_rows + off_a) : 0;
    const int32_t row_b = off_b < o_end ? __ldca(a.dst_rows + off_b) : 0;
    float dpart[8], rpart[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) dpart[q] = rpart[q] = 0.0f;
    // start of destination j's rows, j in [0, kTask] (o_end from nv on)
    auto off_of = [&](int j) -> int32_t {
      const int32_t x = __shfl_sync(0xffffffffu, j < 8 ? off_a : off_b, j & 7, 8);
      return j >= nv ? o_end : x;
    };
    auto first_row = [&](int j, bool some) -> Row8 {  // zeros if it has none
      const int32_t r = __shfl_sync(0xffffffffu, j < 8 ? row_a : row_b, j & 7, 8);
      Row8 x = {{0, 0, 0, 0}};
      if (some) x = load_row(a.interm + (int64_t)r * kCols + lane8 * 8);
      return x;
    };
    // the first rows of the next two destinations are on their way
    int32_t o0 = off_of(0), o1 = off_of(1), o2 = off_of(2);
    Row8 ahead[2] = {first_row(0, o0 < o1), first_row(1, o1 < o2)};
#pragma unroll 2
    for (int j = 0; j < kTask; ++j) {  // a warp's octets go through their destinations together
      Row8 sum = ahead[j & 1];
      const int32_t p0 = o0 + 1, p1 = o1;
      const int32_t o3 = off_of(min(j + 3, kTask));
      if (j + 2 < kTask) ahead[j & 1] = first_row(j + 2, o2 < o3);
      o0 = o1; o1 = o2; o2 = o3;
      const float iv = __shfl_sync(0xffffffffu, j < 8 ? inv_a : inv_b, j & 7, 8);
      if (j >= nv) continue;
      for (int32_t p = p0; p < p1; p += 2) {
        const int32_t r0 = __ldca(a.dst_rows + p), r1 = p + 1 < p1 ? __ldca(a.dst_rows + p + 1) : 0;
        const Row8 x = load_row(a.interm + (int64_t)r0 * kCols + lane8 * 8);
        Row8 y = {{0, 0, 0, 0}};
        if (p + 1 < p1) y = load_row(a.interm + (int64_t)r1 * kCols + lane8 * 8);
        add_row(sum, x);
        if (p + 1 < p1) add_row(sum, y);
      }
      const int64_t v = v0 + j;
      float r[8];
      unpack(sum, r);
#pragma unroll
      for (int q = 0; q < 8; ++q) r[q] *= a.d;
      if ((sbits >> j) & 1u) {
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (s_seed[lane8 * 8 + q] == (int32_t)v) r[q] += s_tele[lane8 * 8 + q];
      }
      if (iv != 0.0f) {
        float c[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) c[q] = r[q] * iv;
        store_contrib<PLANES>(a.contrib, v, lane8, c);
      } else {
#pragma unroll
        for (int q = 0; q < 8; ++q) dpart[q] += r[q];
      }
      if (a.r_out) {  // the caller's: 16-byte aligned
        float4* p = reinterpret_cast<float4*>(a.r_out + v * kCols + lane8 * 8);
        __stcs(p, make_float4(r[0], r[1], r[2], r[3]));
        __stcs(p + 1, make_float4(r[4], r[5], r[6], r[7]));
      }
      if (RESID) {
        const float4* p = reinterpret_cast<const float4*>(a.r_old + v * kCols + lane8 * 8);
        const float4 x = __ldcs(p), y = __ldcs(p + 1);
        const float o[8] = {x.x, x.y, x.z, x.w, y.x, y.y, y.z, y.w};
#pragma unroll
        for (int q = 0; q < 8; ++q) rpart[q] += fabsf(r[q] - o[q]);
      }
    }
    // (FP64 adds run at 2 per cycle and SM: most tasks have no dangling mass)
    bool any = false;
#pragma unroll
    for (int q = 0; q < 8; ++q) any = any || dpart[q] != 0.0f;
    if (any) {
#pragma unroll
      for (int q = 0; q < 8; ++q) s_acc[w][0][q][lane] += (double)dpart[q];
    }
    if (RESID) {
#pragma unroll
      for (int q = 0; q < 8; ++q) s_acc[w][RESID][q][lane] += (double)rpart[q];
    }
  }
  // per-column partials: octets of a warp, then warps of the block
  __syncthreads();
  if (threadIdx.x < 2 * kCols) {
    const int which = threadIdx.x / kCols, j = threadIdx.x % kCols;
    double s = 0.0;
    if (which == 0 || RESID)
      for (int q = 0; q < kThreads / 32; ++q)
        for (int o = 0; o < 4; ++o) s += s_acc[q][RESID ? which : 0][j & 7][8 * o + (j >> 3)];
    a.partials[(int64_t)blockIdx.x * 2 * kCols + threadIdx.x] = s;
  }
  // the last block of 32 adds up their sums, the last of those the groups': a
  // fixed order, 8 loads in flight per thread (one block adding up all 608
  // one after the other took 40 us)
  const int group = blockIdx.x / kMergeGroup, ngroups = (gridDim.x + kMergeGroup - 1) / kMergeGroup;
  const int size = min(kMergeGroup, (int)gridDim.x - group * kMergeGroup);
  double* gsum = a.partials + (int64_t)gridDim.x * 2 * kCols;
  auto add_up = [&](const double* src, int n) -> double {  // valid in threads < 2 kCols
    constexpr int U = 8;
    const int j = threadIdx.x % (2 * kCols), half = threadIdx.x / (2 * kCols);
    double s = 0.0;
#pragma unroll 1
    for (int b0 = 0; b0 < n; b0 += 2 * U) {
      double x[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int b = b0 + 2 * u + half;
        x[u] = b < n ? __ldcg(src + (int64_t)b * 2 * kCols + j) : 0.0;
      }
#pragma unroll
      for (int u = 0; u < U; ++u) s += x[u];
    }
    __syncthreads();
    if (half == 1) s_half[j] = s;
    __syncthreads();
    return half == 0 ? s + s_half[j] : 0.0;
  };
  auto last_of = [&](unsigned* count, int n) -> bool {
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = atomicAdd(count, 1u) == (unsigned)n - 1;
    __syncthreads();
    const bool last = s_last;
    if (last) __threadfence();
    return last;
  };
  if (!last_of(a.counter + 1 + group, size)) return;
  double s = add_up(a.partials + (int64_t)group * kMergeGroup * 2 * kCols, size);
  if (threadIdx.x < 2 * kCols) gsum[(int64_t)group * 2 * kCols + threadIdx.x] = s;
  if (threadIdx.x == 0) a.counter[1 + group] = 0u;
  if (!last_of(a.counter, ngroups)) return;
  s = add_up(gsum, ngroups);
  if (threadIdx.x < kCols) a.D[threadIdx.x] = s;
  else if (RESID && a.resid && threadIdx.x < 2 * kCols) a.resid[threadIdx.x - kCols] = s;
  if (threadIdx.x == 0) *a.counter = 0u;
}

// ---------------------------------------------------------------------------
// Set-up kernels
// ---------------------------------------------------------------------------
__global__ void ppr_chunks_kernel(const int32_t* __restrict__ rp, const int64_t* __restrict__ meta,
                                  const PprSeg* __restrict__ segs, int k, int64_t nchunks,
                                  int2* __restrict__ chunks) {
  // meta: row_base[k+1], edge_base[k+1] of the segmented graph
  const int64_t* row_base = meta;
  const int64_t* edge_base = meta + (k + 1);
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    int s0 = 0, s1 = k;  // last segment with chunk0 <= c (and edges)
    while (s1 - s0 > 1) {
      const int mid = (s0 + s1) >> 1;
      if (segs[mid].chunk0 <= c) s0 = mid; else s1 = mid;
    }
    while (s0 + 1 < k && segs[s0 + 1].chunk0 <= c) ++s0;
    const int64_t e = edge_base[s0] + (c - segs[s0].chunk0) * kChunk;
    int64_t lo = row_base[s0], hi = row_base[s0 + 1];  // last row with rp[row] <= e
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (rp[mid] <= e) lo = mid + 1; else hi = mid;
    }
    chunks[c] = make_int2((int32_t)(lo - 1), s0);
  }
}

// The row open at each chunk's end (-1 when the chunk ends a row): the
// subgraph row of the chunk's last edge, if that row continues past it.
__global__ void carry_rows_kernel(const int32_t* __restrict__ rp, const int64_t* __restrict__ meta,
                                  const PprSeg* __restrict__ segs, const int2* __restrict__ chunks,
                                  int k, int64_t nchunks, int32_t* __restrict__ carry_row) {
  const int64_t* row_base = meta;
  const int64_t* edge_base = meta + (k + 1);
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < nchunks;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int s = chunks[c].y;
    const int64_t el = (c - segs[s].chunk0) * kChunk;
    const int64_t n = min((int64_t)kChunk, (int64_t)segs[s].E - el);
    const int64_t e = edge_base[s] + el + n - 1;  // global index of the chunk's last edge
    int64_t lo = row_base[s], hi = row_base[s + 1];  // last row with rp[row] <= e
    while (lo < hi) {
      const int64_t mid = (lo + hi) >> 1;
      if (rp[mid] <= e) lo = mid + 1; else hi = mid;
    }
    const int64_t row = lo - 1;
    carry_row[c] = (int64_t)rp[row + 1] - 1 > e ? (int32_t)row : -1;
  }
}

__global__ void count_dst_kernel(const int32_t* __restrict__ idx_map, int64_t rows,
                                 int32_t* __restrict__ cnt) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x)
    atomicAdd(cnt + idx_map[r], 1);
}

__global__ void narrow_kernel(const int64_t* __restrict__ in, int64_t n, int32_t* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    out[i] = (int32_t)in[i];
}

// Rows of one segment: their destinations are distinct, so each takes the
// next free slot of its destination's list without collisions; segments
// are filled in order, so every list is in segment order.
__global__ void fill_dst_kernel(const int32_t* __restrict__ idx_map, int64_t r0, int64_t r1,
                                const int32_t* __restrict__ off, int32_t* __restrict__ fill,
                                int32_t* __restrict__ dst_rows) {
  for (int64_t r = r0 + (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < r1;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t v = idx_map[r];
    dst_rows[off[v] + fill[v]] = (int32_t)r;
    fill[v] += 1;
  }
}

__global__ void ppr_seed_kernel(const float* __restrict__ inv, const int32_t* __restrict__ seeds,
                                void* __restrict__ contrib, int planes,
                                uint32_t* __restrict__ seed_bits, double* __restrict__ D) {
  const int j = threadIdx.x;
  if (j >= kCols) return;
  const int32_t s = seeds[j];
  const float c = inv[s];  // R_0 = one-hot at the seed: C = 1 / outdeg
  if (planes == 2)
    static_cast<float*>(contrib)[(int64_t)s * kCols + j] = c;
  else
    static_cast<__nv_bfloat16*>(contrib)[(int64_t)s * kCols + j] = __float2bfloat16_rn(c);
  atomicOr(seed_bits + (s >> 5), 1u << (s & 31));
  D[j] = c == 0.0f ? 1.0 : 0.0;
}

int merge_launch(cg_ppr* p, const float* inv, double damping, float* r_out, const float* r_old,
                 double* resid, cudaStream_t s) {
  MergeArgs a;
  a.dst_off = p->dst_off;
  a.dst_rows = p->dst_rows;
  a.interm = p->interm;
  a.inv = inv;
  a.seeds = p->seeds;
  a.seed_bits = p->seed_bits;
  a.contrib = p->contrib;
  a.r_out = r_out;
  a.r_old = r_old;
  a.D = p->D;
  a.resid = resid;
  a.partials = p->partials;
  a.counter = p->counter;
  a.d = (float)damping;
  a.V = p->V;
  const bool res = r_old != nullptr;
  auto fn = p->planes == 2 ? (res ? ppr_merge_kernel<2, true> : ppr_merge_kernel<2, false>)
                           : (res ? ppr_merge_kernel<1, true> : ppr_merge_kernel<1, false>);
  return launch_chained(fn, p->merge_grid, kThreads, 0, s, a);
}

int gather_launch(cg_ppr* p, cudaStream_t s) {
  if (p->nchunks == 0) return CG_OK;
  const SegPlan& sp = p->seg->plan;
  return launch_chained(p->planes == 2 ? ppr_gather_kernel<2> : ppr_gather_kernel<1>,
                        p->gather_grid, kThreads, 0, s, sp.colf, p->segs, p->chunks, p->nchunks,
                        p->contrib, p->interm, p->carry);
}

int fixup_launch(cg_ppr* p, cudaStream_t s) {
  if (p->npieces == 0) return CG_OK;
  return launch_chained(ppr_fixup_kernel, grid_for(p->npieces * 8, kThreads, 8), kThreads, 0, s,
                        p->pieces, p->npieces, p->runs, p->carry, p->piece_sum, p->run_done,
                        p->interm);
}

void ppr_free(cg_ppr* p) {
  ppr_dense_free(p);
  cudaFree(p->segs);
  cudaFree(p->chunks);
  cudaFree(p->carry);
  cudaFree(p->pieces);
  cudaFree(p->runs);
  cudaFree(p->piece_sum);
  cudaFree(p->run_done);
  cudaFree(p->dst_off);
  cudaFree(p->dst_rows);
  cudaFree(p->interm);
  cudaFree(p->contrib);
  cudaFree(p->r_prev);
  cudaFree(p->seeds);
  cudaFree(p->seed_bits);
  cudaFree(p->D);
  cudaFree(p->partials);
  cudaFree(p->counter);
  delete p;
}

template <class T>
cudaError_t alloc(T** ptr, int64_t n, int64_t* total) {
  const size_t b = sizeof(T) * (size_t)(n > 0 ? n : 1);
  *total += (int64_t)b;
  return cudaMalloc((void**)ptr, b);
}

int ppr_build(cg_ppr* p, cudaStream_t s) {
  const cg_segmented* g = p->seg;
  const SegPlan& sp = g->plan;
  const int k = g->k;
  int64_t& B = p->bytes;
  // segment table and gather chunks
  std::vector<PprSeg> hs(k > 0 ? k : 1);
  int64_t nch = 0;
  for (int q = 0; q < k; ++q) {
    hs[q].cstart = sp.h_cstart[q];
    hs[q].chunk0 = nch;
    hs[q].lo = (int32_t)sp.src_bounds[q];
    hs[q].E = (int32_t)(sp.edge_base[q + 1] - sp.edge_base[q]);
    nch += ceil_div(hs[q].E, kChunk);
  }
  p->nchunks = nch;
  CG_CUDA(alloc(&p->segs, k, &B));
  CG_CUDA(cudaMemcpyAsync(p->segs, hs.data(), sizeof(PprSeg) * k, cudaMemcpyHostToDevice, s));
  CG_CUDA(alloc(&p->chunks, nch, &B));
  CG_CUDA(alloc(&p->carry, nch * kCols, &B));
  if (nch > 0) {
    ppr_chunks_kernel<<<grid_for(nch, 256), 256, 0, s>>>(sp.rp32, sp.meta, p->segs, k, nch,
                                                          p->chunks);
    CG_LAUNCH_CHECK();
    // runs of carries (static) cut into pieces
    int32_t* crow = nullptr;
    CG_CUDA(cudaMallocAsync((void**)&crow, sizeof(int32_t) * (size_t)nch, s));
    carry_rows_kernel<<<grid_for(nch, 256), 256, 0, s>>>(sp.rp32, sp.meta, p->segs, p->chunks,
                                                         k, nch, crow);
    cudaError_t ce = cudaGetLastError();
    std::vector<int32_t> hc((size_t)nch);
    if (ce == cudaSuccess)
      ce = cudaMemcpyAsync(hc.data(), crow, sizeof(int32_t) * (size_t)nch,
                           cudaMemcpyDeviceToHost, s);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(s);
    cudaFreeAsync(crow, s);
    if (ce != cudaSuccess) return cuda_fail(ce, "ppr_batched_create", __FILE__, __LINE__);
    std::vector<int4> hp, hr;
    for (int64_t c = 0; c < nch;) {
      if (hc[c] < 0) { ++c; continue; }
      int64_t e = c + 1;
      while (e < nch && hc[e] == hc[c]) ++e;
      const int32_t run = (int32_t)hr.size(), p0 = (int32_t)hp.size();
      for (int64_t x = c; x < e; x += kPprPiece)
        hp.push_back(make_int4((int32_t)x, (int32_t)std::min<int64_t>(kPprPiece, e - x), run, 0));
      hr.push_back(make_int4(hc[c], p0, (int32_t)hp.size() - p0, 0));
      c = e;
    }
    p->npieces = (int64_t)hp.size();
    p->nruns = (int64_t)hr.size();
    CG_CUDA(alloc(&p->pieces, p->npieces, &B));
    CG_CUDA(alloc(&p->runs, p->nruns, &B));
    CG_CUDA(alloc(&p->piece_sum, p->npieces * kCols, &B));
    CG_CUDA(alloc(&p->run_done, p->nruns, &B));
    if (p->npieces > 0) {
      CG_CUDA(cudaMemcpyAsync(p->pieces, hp.data(), sizeof(int4) * hp.size(),
                              cudaMemcpyHostToDevice, s));
      CG_CUDA(cudaMemcpyAsync(p->runs, hr.data(), sizeof(int4) * hr.size(),
                              cudaMemcpyHostToDevice, s));
      CG_CUDA(cudaMemsetAsync(p->run_done, 0, sizeof(unsigned) * hr.size(), s));
      CG_CUDA(cudaStreamSynchronize(s));  // hp / hr go out of scope
    }
  }
  // destination-major row lists
  const int32_t V = p->V;
  int32_t* cnt = nullptr;
  int64_t* off64 = nullptr;
  CG_CUDA(alloc(&p->dst_off, (int64_t)V + 1, &B));
  CG_CUDA(alloc(&p->dst_rows, p->rows, &B));
  CG_CUDA(cudaMallocAsync((void**)&cnt, sizeof(int32_t) * (size_t)V, s));
  cudaError_t e = cudaMallocAsync((void**)&off64, sizeof(int64_t) * ((size_t)V + 1), s);
  int st = CG_OK;
  if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)V, s);
  if (e == cudaSuccess && p->rows > 0) {
    count_dst_kernel<<<grid_for(p->rows, 256), 256, 0, s>>>(g->idx_map, p->rows, cnt);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) st = exclusive_scan_i32_to_i64(cnt, off64, V, s);
  if (e == cudaSuccess && st == CG_OK) {
    narrow_kernel<<<grid_for((int64_t)V + 1, 256), 256, 0, s>>>(off64, (int64_t)V + 1, p->dst_off);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess && st == CG_OK) e = cudaMemsetAsync(cnt, 0, sizeof(int32_t) * (size_t)V, s);
  for (int q = 0; q < k && e == cudaSuccess && st == CG_OK; ++q) {
    const int64_t r0 = g->row_base[q], r1 = g->row_base[q + 1];
    if (r1 > r0) {
      fill_dst_kernel<<<grid_for(r1 - r0, 256), 256, 0, s>>>(g->idx_map, r0, r1, p->dst_off, cnt,
                                                              p->dst_rows);
      e = cudaGetLastError();
    }
  }
  cudaFreeAsync(cnt, s);
  cudaFreeAsync(off64, s);
  if (st != CG_OK) return st;
  if (e != cudaSuccess) return cuda_fail(e, "ppr_batched_create", __FILE__, __LINE__);
  // iteration state
  CG_CUDA(alloc(&p->interm, p->rows * kCols, &B));
  CG_CUDA(alloc(&p->contrib, (int64_t)V * 8 * p->planes, &B));
  CG_CUDA(alloc(&p->r_prev, (int64_t)V * kCols, &B));
  CG_CUDA(alloc(&p->seeds, kCols, &B));
  CG_CUDA(alloc(&p->seed_bits, ceil_div(V, 32), &B));
  CG_CUDA(alloc(&p->D, kCols, &B));
  // launch shapes: whole waves of resident blocks
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  int per_sm = 0;
  CG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, p->planes == 2 ? ppr_merge_kernel<2, true> : ppr_merge_kernel<1, true>, kThreads,
      0));
  p->merge_grid = di.sm_count * (per_sm > 0 ? per_sm : 1);
  CG_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
      &per_sm, p->planes == 2 ? ppr_gather_kernel<2> : ppr_gather_kernel<1>, kThreads, 0));
  p->gather_grid = di.sm_count * (per_sm > 0 ? per_sm : 1);
  const int64_t groups = ceil_div(p->merge_grid, kMergeGroup);
  CG_CUDA(alloc(&p->partials, (p->merge_grid + groups) * 2 * kCols, &B));
  CG_CUDA(alloc(&p->counter, 1 + groups, &B));
  CG_CUDA(cudaMemsetAsync(p->counter, 0, sizeof(unsigned) * (size_t)(1 + groups), s));
  CG_CUDA(cudaStreamSynchronize(s));
  return CG_OK;
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int ppr_batched_create(const cg_segmented* seg, int32_t planes, cg_ppr** out,
                       cudaStream_t stream) {
  CG_ARG(out != nullptr, "ppr_batched_create: out is NULL");
  *out = nullptr;
  CG_ARG(seg != nullptr, "ppr_batched_create: null segmented graph");
  CG_ARG(planes == 1 || planes == 2, "ppr_batched_create: planes must be 1 or 2 (got %d)",
         planes);
  int dev = 0;
  CG_CUDA(cudaGetDevice(&dev));
  CG_ARG(dev == seg->device, "ppr_batched_create: the segmented graph lives on device %d, "
         "current device is %d", seg->device, dev);
  cg_ppr* p = new cg_ppr();
  p->device = dev;
  p->seg = seg;
  p->V = seg->V;
  p->k = seg->k;
  p->rows = seg->rows;
  p->planes = planes;
  const int st = ppr_build(p, stream);
  if (st != CG_OK) {
    cudaStreamSynchronize(stream);
    ppr_free(p);
    return st;
  }
  *out = p;
  return CG_OK;
}

int ppr_batched_destroy(cg_ppr* p) {
  if (!p) return CG_OK;
  cudaDeviceSynchronize();
  ppr_free(p);
  return CG_OK;
}

int ppr_batched_bytes(const cg_ppr* p, int64_t* bytes, int64_t* chunks) {
  CG_ARG(p != nullptr, "ppr_batched_bytes: null handle");
  if (bytes) *bytes = p->bytes;
  if (chunks) *chunks = p->nchunks;
  return CG_OK;
}

int ppr_batched_init(cg_ppr* p, const float* inv, const int32_t* host_seeds,
                     cudaStream_t stream) {
  CG_ARG(p && inv && host_seeds, "ppr_batched_init: null argument");
  for (int j = 0; j < kCols; ++j)
    CG_ARG(host_seeds[j] >= 0 && host_seeds[j] < p->V,
           "ppr_batched_init: seed %d of column %d outside [0, %d)", host_seeds[j], j, p->V);
  CG_CUDA(cudaMemcpyAsync(p->seeds, host_seeds, sizeof(int32_t) * kCols, cudaMemcpyHostToDevice,
                          stream));
  CG_CUDA(cudaMemsetAsync(p->contrib, 0, sizeof(uint4) * 8 * p->planes * (size_t)p->V, stream));
  CG_CUDA(cudaMemsetAsync(p->seed_bits, 0, sizeof(uint32_t) * (size_t)ceil_div(p->V, 32),
                          stream));
  ppr_seed_kernel<<<1, kCols, 0, stream>>>(inv, p->seeds, p->contrib, p->planes, p->seed_bits,
                                           p->D);
  CG_LAUNCH_CHECK();
  CG_TRY(ppr_dense_pack(p, stream));
  // host_seeds may go out of scope on return
  CG_CUDA(cudaStreamSynchronize(stream));
  p->seeded = true;
  return CG_OK;
}

int ppr_batched_step(cg_ppr* p, const float* inv, double damping, int32_t phases,
                     const float* rank_old, float* rank_out, double* resid,
                     cudaStream_t stream) {
  CG_ARG(p && inv, "ppr_batched_step: null argument");
  CG_ARG(p->seeded, "ppr_batched_step: call ppr_batched_init first");
  CG_ARG(damping >= 0.0 && damping <= 1.0, "ppr_batched_step: damping must be in [0, 1]");
  CG_ARG(phases >= 0 && phases <= 15, "ppr_batched_step: phases must be in [0, 15]");
  CG_ARG(!resid || rank_old, "ppr_batched_step: the residual needs rank_old");
  CG_ARG(!rank_old || rank_out, "ppr_batched_step: rank_old needs rank_out");
  CG_ARG(!rank_out || (const float*)rank_out != rank_old,
         "ppr_batched_step: rank_out must not alias rank_old");
  if (phases & 1) CG_TRY(gather_launch(p, stream));
  if (phases & 8) CG_TRY(ppr_dense_launch(p, stream));  // the hub block's rows (if attached)
  if (phases & 2) CG_TRY(fixup_launch(p, stream));
  if (phases & 4) {
    CG_TRY(merge_launch(p, inv, damping, rank_out, rank_old, resid, stream));
    CG_TRY(ppr_dense_pack(p, stream));
  }
  return CG_OK;
}

int ppr_batched_iterate(cg_ppr* p, const float* inv, double damping, int32_t iterations,
                        float* rank_out, double* resid, cudaStream_t stream) {
  CG_ARG(p && inv, "ppr_batched_iterate: null argument");
  CG_ARG(iterations >= 1, "ppr_batched_iterate: iterations must be >= 1");
  CG_ARG(!resid || (iterations >= 2 && rank_out),
         "ppr_batched_iterate: the residual needs iterations >= 2 and rank_out");
  for (int t = 0; t < iterations; ++t) {
    const bool last = t == iterations - 1;
    const bool before_last = t == iterations - 2 && resid;
    float* r_out = last ? rank_out : before_last ? p->r_prev : nullptr;
    const float* r_old = last && resid ? p->r_prev : nullptr;
    CG_TRY(ppr_batched_step(p, inv, damping, 15, r_old, r_out, last ? resid : nullptr, stream));
  }
  return CG_OK;
}

}  // extern "C"
