// The collaborative-filtering gather: for every rating the neighbour's factor
// row, its product with the vertex's own, and the error's share of the gradient.
//
// What bounds it is the rows' way from L2: 128 bytes per rating (K = 32, 32-bit
// entries) at 64 bytes per cycle and SM, 0.68 ms per side for 99 M ratings at
// 1.92 GHz; the gathers take 0.79 and 0.82 ms.  Everything else is kept out of
// its way:
//   pieces  consecutive ratings of one vertex, LANES lanes per piece, 32 / LANES
//           pieces in a warp's task, sorted by length so that those of a task are
//           about equally long.  A group's gradient needs no reduction over the
//           warp, and a row is one 32-byte read per lane.
//   sums    four ratings at a time: packed FMAs, and one reduction that leaves
//           each lane of four with one rating's product (104 instructions per
//           32 ratings at K = 32).
//   rows    are not kept in L1 (K = 32 users, whose 17,770 items fit in L2 many
//           times over: 0.91 -> 0.79 ms); 20 warps per SM with four rows per group in
//           flight (24 gain on one side what they lose on the other, 16: 0.94 and
//           0.95 ms, 32 spill: 1.39 and 1.12).
// Before, 99 M ratings at K = 32, hi + lo: a warp per piece, a row read in two
// parts and unpacked from BF16 pairs, 1.61 and 1.27 ms; rows in shared memory, a
// segment of them at a time, 1.06 and 1.01 ms, and 0.31 ms instead of 0.06 for the
// updates, whose partial gradients were ten times as many.
#include <algorithm>

#include <cuda_bf16.h>

#include "cf_rows.cuh"

namespace cg {
namespace {

constexpr int kRowThreads = 128;  // threads per gather block
constexpr int kLongest = 256;     // ratings per piece at most (sort keys: 8 bits)
constexpr int kShortest = 16;

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
__device__ __forceinline__ u64 bf2(uint32_t w) {
  return (u64)(w & 0xffff0000u) << 32 | (w << 16);
}

// A lane's EL dimensions of a row, as FP32 pairs: row-long reads of a lane group.
template <bool BF16, int EL>
struct RowPart {
  u64 p[EL / 2];
  __device__ __forceinline__ void zero() {
#pragma unroll
    for (int q = 0; q < EL / 2; ++q) p[q] = 0ull;
  }
  __device__ __forceinline__ void load(const char* at) {
    if constexpr (BF16) {
      if constexpr (EL == 8) {
        uint32_t a, b, c, d;
        asm volatile("ld.global.v4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "l"(at));
        p[0] = bf2(a); p[1] = bf2(b); p[2] = bf2(c); p[3] = bf2(d);
      } else {
        uint32_t a, b;
        asm volatile("ld.global.v2.b32 {%0, %1}, [%2];" : "=r"(a), "=r"(b) : "l"(at));
        p[0] = bf2(a); p[1] = bf2(b);
      }
    } else if constexpr (EL == 8) {
      asm volatile("ld.global.L1::no_allocate.v4.b64 {%0, %1, %2, %3}, [%4];"
                   : "=l"(p[0]), "=l"(p[1]), "=l"(p[2]), "=l"(p[3]) : "l"(at));
    } else {
      asm volatile("ld.global.v2.b64 {%0, %1}, [%2];" : "=l"(p[0]), "=l"(p[1]) : "l"(at));
    }
  }
};

// lanes per rating; gather blocks per SM, by the registers of a lane's parts of
// five rows (K = 16: 8 blocks 3.03 ms for 20 M ratings, 5 blocks 3.42)
template <int K> struct Lanes {
  static constexpr int n = K == 64 ? 8 : 4, kBlocks = K == 16 ? 8 : 5;
};
int pieces_per_task(int K) { return K == 64 ? 4 : 8; }
int blocks_per_sm(int K) { return K == 16 ? Lanes<16>::kBlocks : Lanes<32>::kBlocks; }

template <int K, bool BF16, bool SSE>
__global__ void __launch_bounds__(kRowThreads, Lanes<K>::kBlocks)
cf_rows_kernel(const int4* recs, int32_t ntasks, int32_t nn,
               const int32_t* nbr, const uint8_t* rate,
               const void* self, const void* other,
               float* gpart, double* partials,
               unsigned* counter, double* sse_out) {
  constexpr unsigned kFull = 0xffffffffu;
  constexpr int LANES = Lanes<K>::n, EL = K / LANES, NP = EL / 2, G = 32 / LANES;
  constexpr int kRow = K * (BF16 ? 2 : 4), kPart = EL * (BF16 ? 2 : 4);
  if (!chain_begin()) return;
  const int lane = threadIdx.x & 31, sub = lane % LANES, grp = lane / LANES;
  const int first = lane & ~(LANES - 1);
  const char* mine = static_cast<const char*>(self) + sub * kPart;
  const char* rows = static_cast<const char*>(other) + sub * kPart;
  const int nw = (int)((gridDim.x * blockDim.x) >> 5);
  double se = 0.0;  // squared errors: FP32 within a piece, FP64 over the pieces
  for (int32_t task = (int32_t)((blockIdx.x * blockDim.x + threadIdx.x) >> 5); task < ntasks;
       task += nw) {
    const int64_t slot = (int64_t)task * G + grp;
    const int4 rec = __ldca(recs + slot);
    const int64_t at = (int64_t)(((u64)(uint32_t)rec.y << 32) | (uint32_t)rec.x);
    const int len = rec.z;
    const int32_t* nb = nbr + at + sub;
    const uint8_t* rt = rate + at + sub;
    RowPart<BF16, EL> x;
    u64 g[NP];
    x.zero();
    if (len > 0) x.load(mine + (int64_t)rec.w * kRow);
#pragma unroll
    for (int q = 0; q < NP; ++q) g[q] = 0ull;
    uint32_t un = 0, rn = 0, um = 0, rm = 0;  // this chunk's rating and the next one's
    if (sub < len) {
      un = (uint32_t)*nb;
      rn = *rt;
    }
    if (sub + LANES < len) {
      um = (uint32_t)nb[LANES];
      rm = rt[LANES];
    }
    float te2 = 0.0f;
    const int longest = __shfl_sync(kFull, len, 0);
    for (int c = 0; c < longest; c += LANES) {
      const uint32_t row = min(un, (uint32_t)nn - 1u);
      // the rating as FP32 (2^23 + r without its leading one)
      const float r = __uint_as_float(0x4B000000u | rn) - 8388608.0f;
      const bool real = c + sub < len;
      un = um;
      rn = rm;
      if (c + 2 * LANES + sub < len) {
        um = (uint32_t)nb[c + 2 * LANES];
        rm = rt[c + 2 * LANES];
      }
#pragma unroll
      for (int h = 0; h < LANES; h += 4) {  // four ratings of the group at a time
        RowPart<BF16, EL> y[4];
        float d[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const uint32_t w = __shfl_sync(kFull, row, first + h + j);
          y[j].zero();
          if (c + h + j < len) y[j].load(rows + (int64_t)w * kRow);
        }
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          u64 a = mul2(x.p[0], y[j].p[0]);
#pragma unroll
          for (int q = 1; q < NP; ++q) fma2(a, x.p[q], y[j].p[q]);
          d[j] = halves(a);
        }
        // the group's lanes add their parts and share the four ratings out:
        // lane sub ends up with the product of rating h + (sub & 3)
        const bool o1 = sub & 1, o2 = sub & 2;
        const float a01 = (o1 ? d[1] : d[0]) + __shfl_xor_sync(kFull, o1 ? d[0] : d[1], 1);
        const float a23 = (o1 ? d[3] : d[2]) + __shfl_xor_sync(kFull, o1 ? d[2] : d[3], 1);
        float dot = (o2 ? a23 : a01) + __shfl_xor_sync(kFull, o2 ? a01 : a23, 2);
        if (LANES == 8) dot += __shfl_xor_sync(kFull, dot, 4);
        const float e = real ? r - dot : 0.0f;  // (8 lanes: those of h .. h + 3 hold these)
        if (SSE && (LANES == 4 || (sub & 4) == h)) te2 = fmaf(e, e, te2);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float ej = __shfl_sync(kFull, e, first + h + j);
          const u64 e2 = pair(ej, ej);
#pragma unroll
          for (int q = 0; q < NP; ++q) fma2(g[q], e2, y[j].p[q]);
        }
      }
    }
    if (len > 0) {
      float* dst = gpart + slot * K + sub * EL;
#pragma unroll
      for (int q = 0; q < NP; q += 2)
        __stcs(reinterpret_cast<ulonglong2*>(dst + 2 * q), make_ulonglong2(g[q], g[q + 1]));
    }
    if (SSE) se += (double)te2;
  }
  if (!SSE) return;
  __shared__ double sh[32];
  __shared__ bool s_last;
  const double bs = block_sum<double, kRowThreads>(se, sh);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = bs;
    __threadfence();
    s_last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  double total = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += kRowThreads) total += __ldcg(partials + i);
  total = block_sum<double, kRowThreads>(total, sh);
  if (threadIdx.x == 0) {
    if (sse_out) *sse_out = total;
    *counter = 0u;
  }
}

// ---------------------------------------------------------------------------
// Building the pieces
// ---------------------------------------------------------------------------
__global__ void piece_count_kernel(const int64_t* __restrict__ off, int64_t n, int most,
                                   int64_t* __restrict__ cnt) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x)
    cnt[v] = (off[v + 1] - off[v] + most - 1) / most;
}

// Sort keys (longest first) and vertices of the pieces: one warp per vertex.
__global__ void piece_key_kernel(const int64_t* __restrict__ off, const int64_t* __restrict__ poff,
                                 int64_t n, int most, uint32_t* __restrict__ key,
                                 int32_t* __restrict__ item, int32_t* __restrict__ vtx) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; v < n; v += nw) {
    const int64_t p0 = poff[v], p1 = poff[v + 1], deg = off[v + 1] - off[v];
    for (int64_t p = p0 + lane; p < p1; p += 32) {
      const int64_t left = deg - (p - p0) * most;
      key[p] = (uint32_t)(most - (left < most ? left : most));
      item[p] = (int32_t)p;
      vtx[p] = (int32_t)v;
    }
  }
}

__global__ void piece_slot_kernel(const int32_t* __restrict__ order, const int32_t* __restrict__ vtx,
                                  const int64_t* __restrict__ off, const int64_t* __restrict__ poff,
                                  int64_t npieces, int64_t nslots, int most, int4* __restrict__ recs,
                                  int32_t* __restrict__ slots) {
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nslots;
       q += (int64_t)gridDim.x * blockDim.x) {
    int4 rec = make_int4(0, 0, 0, 0);
    if (q < npieces) {
      const int32_t p = order[q], v = vtx[p];
      const int64_t b = off[v] + (p - poff[v]) * most, left = off[v + 1] - b;
      rec = make_int4((int32_t)(uint32_t)b, (int32_t)(b >> 32), (int)(left < most ? left : most), v);
      slots[p] = (int32_t)q;
    }
    recs[q] = rec;
  }
}

template <int K, bool BF16>
int launch(const CfPieces& c, int64_t nn, const int32_t* nbr, const uint8_t* rate,
           const void* self, const void* other, bool with_sse, double* partials,
           unsigned* counter, double* sse, int grid, cudaStream_t s) {
  return launch_chained(with_sse ? cf_rows_kernel<K, BF16, true> : cf_rows_kernel<K, BF16, false>,
                        grid, kRowThreads, 0, s, c.recs, c.ntasks, nn, nbr, rate, self, other,
                        c.gpart, partials, counter, sse);
}

}  // namespace

int cf_rows_grid(int K, int* grid) {
  DeviceInfo di{};
  CG_TRY(device_info(&di));
  *grid = di.sm_count * blocks_per_sm(K);
  return CG_OK;
}

int cf_rows_gather(const CfPieces& c, int K, bool bf16, int64_t nn, const int32_t* nbr,
                   const uint8_t* rate, const void* self, const void* other, bool with_sse,
                   double* partials, unsigned* counter, double* sse, int grid, cudaStream_t s) {
  if (c.ntasks == 0) {
    if (with_sse && sse) CG_CUDA(cudaMemsetAsync(sse, 0, sizeof(double), s));
    return CG_OK;
  }
  auto run = K == 16 ? (bf16 ? launch<16, true> : launch<16, false>)
             : K == 32 ? (bf16 ? launch<32, true> : launch<32, false>)
                       : (bf16 ? launch<64, true> : launch<64, false>);
  return run(c, nn, nbr, rate, self, other, with_sse, partials, counter, sse, grid, s);
}

int cf_pieces_build(CfPieces* c, int64_t n, int64_t R, int K, const int64_t* off, int few,
                    cudaStream_t s) {
  *c = CfPieces();
  int grid = 0;
  CG_TRY(cf_rows_grid(K, &grid));
  const int G = pieces_per_task(K);
  const int64_t groups = (int64_t)grid * (kRowThreads / 32) * G;
  // pieces so short that every group of lanes on the GPU gets two, where the
  // ratings allow that
  c->most = kLongest;
  while (c->most > kShortest && R < 2 * groups * c->most) c->most /= 2;
  const int64_t bound = n + R / c->most;  // pieces at most
  Scratch tmp(s, Scratch::round(8 * (size_t)n) + Scratch::round(8 * (size_t)(n + 1)) +
                     scan_scratch(n) + 5 * Scratch::round(4 * (size_t)bound) + sort_scratch(bound) +
                     4096);
  int64_t *cnt = nullptr, *poff = nullptr;
  int32_t *item = nullptr, *sitem = nullptr, *vtx = nullptr;
  uint32_t *key = nullptr, *skey = nullptr;
  CG_CUDA(tmp.get(&cnt, n));
  CG_CUDA(tmp.get(&poff, n + 1));
  piece_count_kernel<<<grid_for(n, 256), 256, 0, s>>>(off, n, c->most, cnt);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i64(cnt, poff, n, s, &tmp));
  CG_CUDA(cudaMemcpyAsync(&c->npieces, poff + n, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  const int64_t np = c->npieces;
  c->ntasks = (int32_t)ceil_div(np, G);
  const int64_t nslots = (int64_t)c->ntasks * G;
  c->most_many = (int32_t)(np / few + 1);
  const size_t rb = Scratch::round(16 * (size_t)nslots), sb = Scratch::round(4 * (size_t)np),
               pb = Scratch::round(8 * (size_t)(n + 1)),
               mb = Scratch::round(4 * ((size_t)c->most_many + 2));
  c->bytes = (int64_t)(rb + sb + pb + mb) + 4 * nslots * K;
  CG_CUDA(cudaMalloc((void**)&c->slab, (size_t)c->bytes + 256));
  c->recs = reinterpret_cast<int4*>(c->slab);
  c->slots = reinterpret_cast<int32_t*>(c->slab + rb);
  c->poff = reinterpret_cast<int64_t*>(c->slab + rb + sb);
  c->many = reinterpret_cast<int32_t*>(c->slab + rb + sb + pb);
  c->gpart = reinterpret_cast<float*>(c->slab + rb + sb + pb + mb);
  CG_CUDA(cudaMemcpyAsync(c->poff, poff, 8 * (size_t)(n + 1), cudaMemcpyDeviceToDevice, s));
  // (an update before the first gather only decays the factors)
  CG_CUDA(cudaMemsetAsync(c->gpart, 0, 4 * (size_t)nslots * K, s));
  if (np == 0) return CG_OK;
  CG_CUDA(tmp.get(&key, np));
  CG_CUDA(tmp.get(&skey, np));
  CG_CUDA(tmp.get(&item, np));
  CG_CUDA(tmp.get(&sitem, np));
  CG_CUDA(tmp.get(&vtx, np));
  piece_key_kernel<<<grid_for(n * 32, 256), 256, 0, s>>>(off, poff, n, c->most, key, item, vtx);
  CG_LAUNCH_CHECK();
  CG_TRY(radix_sort_pairs(key, item, skey, sitem, np, 8, s, &tmp));
  piece_slot_kernel<<<grid_for(nslots, 256), 256, 0, s>>>(sitem, vtx, off, poff, np, nslots,
                                                          c->most, c->recs, c->slots);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

void cf_pieces_free(CfPieces* c) {
  cudaFree(c->slab);
  *c = CfPieces();
}

}  // namespace cg
