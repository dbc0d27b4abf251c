// Collaborative filtering by gradient descent (the paper's CF application,
// Section VI / Table III) on a user-item rating graph.  One sweep updates
// both sides from the same old factors (Jacobi):
//   e_ui = r_ui - p_u . q_i
//   p_u += step ((1/deg u) sum_{i in N(u)} e_ui q_i - lambda p_u)
//   q_i += step ((1/deg i) sum_{u in N(i)} e_ui p_u - lambda q_i)
// and reports sum e_ui^2 of the old factors (FP64).
//
// Each side is a per-vertex gather of err * neighbour-row over that side's
// CSR (Algorithm 3's gather with a K-wide row and a dot product per edge).  Both
// factor matrices fit in L2 (Netflix shape: 61 MB of user rows and 2.3 MB of item
// rows in 32 bits, half that in BF16), so the source set is one segment and the
// gather is split only for load balance, into pieces of a vertex's ratings
// (cf_rows.cu).  Piece gradients are summed per vertex, in piece order, by the
// update kernel.
//
// Storage precision of P and Q: 32 bits per entry (FP32; also where the caller
// asks for a BF16 hi + lo pair, whose 32 bits hold less), or BF16; arithmetic is
// FP32, SSE is FP64.
#include <cuda_bf16.h>

#include "cf_rows.cuh"

namespace cg {
// Vertices with more pieces are updated by a warp, with more than kCfWide by a
// block: a reader has four rows in flight, so more than that in one chain is
// time (item side of 2 M ratings at K = 64: 7.9 us so, 9.7 with 16 and 96, 28
// with 24 and 384; of 99 M at K = 32: 25, 25 and 39).
constexpr int kCfWarp = 8;
constexpr int kCfWide = 64;
constexpr int kCfThreads = 256;
}  // namespace cg

struct cg_bipartite {
  int device = 0;
  int64_t U = 0, I = 0, R = 0;
  int32_t K = 32;
  bool bf16 = false;           // storage: BF16, else FP32
  const int64_t* uoff = nullptr;
  const int32_t* uitem = nullptr;
  const uint8_t* urate = nullptr;
  const int64_t* ioff = nullptr;
  const int32_t* iuser = nullptr;
  const uint8_t* irate = nullptr;
  cg::CfPieces side[2];
  // vertices with more than kCfWide pieces, and from the list's end those with
  // more than kCfWarp
  int32_t* wide[2] = {nullptr, nullptr};
  int32_t* warp[2] = {nullptr, nullptr};
  int32_t nwide[2] = {0, 0}, nwarp[2] = {0, 0};
  void* P = nullptr;           // factors; one allocation with Q, partials and counter
  void* Q = nullptr;
  double* partials = nullptr;  // [gather grid] SSE
  unsigned* counter = nullptr;
  int gather_grid = 0;
  int64_t bytes = 0;
};

namespace cg {
namespace {

__device__ __forceinline__ float b_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float b_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

__device__ __forceinline__ uint32_t pk(float a, float b) {
  const __nv_bfloat162 p = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t*>(&p);
}

// 8 consecutive dimensions of row `row` (K per row) in the storage format.
template <bool BF16>
__device__ __forceinline__ void load8(const void* p0, int64_t row, int K, int d0, float (&y)[8]) {
  const int64_t at = row * K + d0;
  if (BF16) {
    const uint4 h = __ldca(reinterpret_cast<const uint4*>(static_cast<const uint16_t*>(p0) + at));
    y[0] = b_lo(h.x); y[1] = b_hi(h.x); y[2] = b_lo(h.y); y[3] = b_hi(h.y);
    y[4] = b_lo(h.z); y[5] = b_hi(h.z); y[6] = b_lo(h.w); y[7] = b_hi(h.w);
  } else {
    const float4* f = reinterpret_cast<const float4*>(static_cast<const float*>(p0) + at);
    const float4 a = __ldca(f), b = __ldca(f + 1);
    y[0] = a.x; y[1] = a.y; y[2] = a.z; y[3] = a.w;
    y[4] = b.x; y[5] = b.y; y[6] = b.z; y[7] = b.w;
  }
}

template <bool BF16>
__device__ __forceinline__ void store8(void* p0, int64_t row, int K, int d0, const float (&x)[8]) {
  const int64_t at = row * K + d0;
  if (BF16) {
    *reinterpret_cast<uint4*>(static_cast<uint16_t*>(p0) + at) =
        make_uint4(pk(x[0], x[1]), pk(x[2], x[3]), pk(x[4], x[5]), pk(x[6], x[7]));
  } else {
    float4* f = reinterpret_cast<float4*>(static_cast<float*>(p0) + at);
    f[0] = make_float4(x[0], x[1], x[2], x[3]);
    f[1] = make_float4(x[4], x[5], x[6], x[7]);
  }
}

// Four pieces' gradients (their slots, -1: none) into g, in order.
template <int K>
__device__ __forceinline__ void add_pieces(const float* gpart, const int32_t (&slot)[4],
                                           int d0, float (&g)[8]) {
  float4 a[4], b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    a[u] = b[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (slot[u] >= 0) {
      const float4* s = reinterpret_cast<const float4*>(gpart + (int64_t)slot[u] * K + d0);
      a[u] = __ldcs(s);
      b[u] = __ldcs(s + 1);
    }
  }
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    g[0] += a[u].x; g[1] += a[u].y; g[2] += a[u].z; g[3] += a[u].w;
    g[4] += b[u].x; g[5] += b[u].y; g[6] += b[u].z; g[7] += b[u].w;
  }
}

// The vertices of a side, by their numbers of pieces.
struct UpdateRows {
  const int64_t* poff;   // first piece of each vertex
  const int32_t* slots;  // where the pieces' gradients lie
  const int64_t* off;    // first rating of each vertex
  int64_t n;
  const int32_t* wide;   // more than kCfWide pieces: a block each
  int32_t nwide;
  const int32_t* warp;   // more than kCfWarp: a warp each
  int32_t nwarp;
  const float* gpart;
  void* x0;
  float lambda, step;
};

// x_v += step (g_v / deg v - lambda x_v), g_v = the sum of v's piece gradients,
// the lanes of vertex v's group holding 8 of its dimensions each.
template <int LANES, bool BF16>
__device__ __forceinline__ void update_vertex(const UpdateRows& a, int64_t v, int d0,
                                              const float (&g)[8]) {
  const int64_t deg = a.off[v + 1] - a.off[v];
  const float inv = deg > 0 ? 1.0f / (float)deg : 0.0f;
  float x[8];
  load8<BF16>(a.x0, v, 8 * LANES, d0, x);
#pragma unroll
  for (int q = 0; q < 8; ++q) x[q] = x[q] + a.step * (g[q] * inv - a.lambda * x[q]);
  store8<BF16>(a.x0, v, 8 * LANES, d0, x);
}

// One launch for all vertices of a side, the longest first: blocks for those
// with many pieces (the block's groups of LANES lanes sum interleaved subsets, a
// fixed-order tree over the groups adds these), then warps (the same within a
// warp), then a group per vertex, in piece order; four pieces' reads in flight
// everywhere.  Deterministic.  (As three launches, one after the other, the item
// side of 99 M ratings took 68 us, as one 39.)
template <int LANES, bool BF16>
__global__ void __launch_bounds__(kCfThreads)
cf_update_kernel(UpdateRows a) {
  constexpr int K = 8 * LANES, U = 4;
  __shared__ __align__(16) float red[kCfThreads / LANES * K];
  if (!chain_begin()) return;
  const int sub = threadIdx.x % LANES, d0 = 8 * sub;
  float g[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) g[q] = 0.0f;
  int32_t slot[U];
  int64_t b = blockIdx.x;
  if (b < a.nwide) {
    constexpr int GROUPS = kCfThreads / LANES;
    const int grp = threadIdx.x / LANES;
    const int32_t v = a.wide[b];
    const int64_t p1 = a.poff[v + 1];
    for (int64_t p = a.poff[v] + grp; p < p1; p += U * GROUPS) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        slot[u] = p + u * GROUPS < p1 ? __ldca(a.slots + p + u * GROUPS) : -1;
      add_pieces<K>(a.gpart, slot, d0, g);
    }
#pragma unroll
    for (int q = 0; q < 8; ++q) red[grp * K + d0 + q] = g[q];
    __syncthreads();
    for (int st = GROUPS / 2; st >= 1; st >>= 1) {
      if (grp < st)
#pragma unroll
        for (int q = 0; q < 8; ++q) red[grp * K + d0 + q] += red[(grp + st) * K + d0 + q];
      __syncthreads();
    }
    if (grp == 0) {
#pragma unroll
      for (int q = 0; q < 8; ++q) g[q] = red[d0 + q];
      update_vertex<LANES, BF16>(a, v, d0, g);
    }
    return;
  }
  b -= a.nwide;
  const int64_t wblocks = (a.nwarp + kCfThreads / 32 - 1) / (kCfThreads / 32);
  if (b < wblocks) {
    constexpr int GROUPS = 32 / LANES;
    const int64_t i = b * (kCfThreads / 32) + (threadIdx.x >> 5);
    if (i >= a.nwarp) return;
    const int grp = (threadIdx.x & 31) / LANES;
    const int32_t v = a.warp[i];
    const int64_t p1 = a.poff[v + 1];
    for (int64_t p = a.poff[v] + grp; p < p1; p += U * GROUPS) {
#pragma unroll
      for (int u = 0; u < U; ++u)
        slot[u] = p + u * GROUPS < p1 ? __ldca(a.slots + p + u * GROUPS) : -1;
      add_pieces<K>(a.gpart, slot, d0, g);
    }
    __syncwarp();
#pragma unroll
    for (int o = LANES; o < 32; o <<= 1)
#pragma unroll
      for (int q = 0; q < 8; ++q) g[q] += __shfl_xor_sync(0xffffffffu, g[q], o);
    if (grp == 0) update_vertex<LANES, BF16>(a, v, d0, g);
    return;
  }
  b -= wblocks;
  const int64_t ng = (gridDim.x - a.nwide - wblocks) * (kCfThreads / LANES);
  for (int64_t v = (b * kCfThreads + threadIdx.x) / LANES; v < a.n; v += ng) {
    const int64_t p0 = a.poff[v], p1 = a.poff[v + 1];
    if (p1 - p0 > kCfWarp) continue;
#pragma unroll
    for (int q = 0; q < 8; ++q) g[q] = 0.0f;
    for (int64_t p = p0; p < p1; p += U) {
#pragma unroll
      for (int u = 0; u < U; ++u) slot[u] = p + u < p1 ? __ldca(a.slots + p + u) : -1;
      add_pieces<K>(a.gpart, slot, d0, g);
    }
    update_vertex<LANES, BF16>(a, v, d0, g);
  }
}

template <int LANES, bool BF16>
__global__ void cf_encode_kernel(const float* __restrict__ in, int64_t n, void* x0) {
  constexpr int K = 8 * LANES;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * LANES;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = t / LANES;
    const int d0 = 8 * (int)(t % LANES);
    float x[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) x[q] = in[v * K + d0 + q];
    store8<BF16>(x0, v, K, d0, x);
  }
}

template <int LANES, bool BF16>
__global__ void cf_decode_kernel(const void* x0, int64_t n,
                                 float* __restrict__ out) {
  constexpr int K = 8 * LANES;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * LANES;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t v = t / LANES;
    const int d0 = 8 * (int)(t % LANES);
    float x[8];
    load8<BF16>(x0, v, K, d0, x);
#pragma unroll
    for (int q = 0; q < 8; ++q) out[v * K + d0 + q] = x[q];
  }
}

// user of every rating of the user-major CSR, and the item keys to sort by
__global__ void expand_users_kernel(const int64_t* __restrict__ uoff, int64_t U,
                                    const int32_t* __restrict__ uitem, int32_t* __restrict__ user,
                                    uint32_t* __restrict__ key, int32_t* __restrict__ idx) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < U; u += nw)
    for (int64_t e = uoff[u] + lane; e < uoff[u + 1]; e += 32) {
      user[e] = (int32_t)u;
      key[e] = (uint32_t)uitem[e];
      idx[e] = (int32_t)e;
    }
}

__global__ void item_hist_kernel(const int32_t* __restrict__ uitem, int64_t R, int64_t I,
                                 int64_t* __restrict__ cnt, int32_t* __restrict__ bad) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < R;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = uitem[e];
    if (i < 0 || i >= I) {
      atomicExch(bad, 1);
      continue;
    }
    atomicAdd(reinterpret_cast<unsigned long long*>(cnt + i), 1ull);
  }
}

__global__ void transpose_gather_kernel(const int32_t* __restrict__ order, int64_t R,
                                        const int32_t* __restrict__ user,
                                        const uint8_t* __restrict__ urate,
                                        int32_t* __restrict__ iuser, uint8_t* __restrict__ irate) {
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < R;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = order[e];
    iuser[e] = user[s];
    irate[e] = urate[s];
  }
}

template <int LANES, bool BF16>
int update_side(cg_bipartite* h, int side, float lambda, float step, cudaStream_t s) {
  const int64_t n = side == 0 ? h->U : h->I;
  const CfPieces& c = h->side[side];
  const UpdateRows a{c.poff, c.slots, side == 0 ? h->uoff : h->ioff, n, h->wide[side],
                     h->nwide[side], h->warp[side], h->nwarp[side], c.gpart,
                     side == 0 ? h->P : h->Q, lambda, step};
  const int64_t blocks = h->nwide[side] + ceil_div(h->nwarp[side], kCfThreads / 32) +
                         grid_for(n * LANES, kCfThreads, 8);
  return launch_chained(cf_update_kernel<LANES, BF16>, (unsigned)blocks, kCfThreads, 0, s, a);
}

template <int LANES>
int update_dispatch(cg_bipartite* h, int side, float lambda, float step, cudaStream_t s) {
  return h->bf16 ? update_side<LANES, true>(h, side, lambda, step, s)
                 : update_side<LANES, false>(h, side, lambda, step, s);
}

// phase: 0 user gather, 1 item gather, 2 user update, 3 item update
int run_phase(cg_bipartite* h, int phase, double* sse, float lambda, float step, cudaStream_t s) {
  const int side = phase & 1;
  if (phase < 2)  // side 0: users gather item rows; side 1: items gather user rows
    return cf_rows_gather(h->side[side], h->K, h->bf16, side == 0 ? h->I : h->U,
                          side == 0 ? h->uitem : h->iuser, side == 0 ? h->urate : h->irate,
                          side == 0 ? h->P : h->Q, side == 0 ? h->Q : h->P, side == 0,
                          h->partials, h->counter, sse, h->gather_grid, s);
  switch (h->K) {
    case 16: return update_dispatch<2>(h, side, lambda, step, s);
    case 32: return update_dispatch<4>(h, side, lambda, step, s);
    default: return update_dispatch<8>(h, side, lambda, step, s);
  }
}

template <int LANES>
int codec(cg_bipartite* h, const float* P, const float* Q, float* Pout, float* Qout,
          cudaStream_t s) {
  const int64_t n[2] = {h->U, h->I};
  void* st[2] = {h->P, h->Q};
  const float* in[2] = {P, Q};
  float* out[2] = {Pout, Qout};
  for (int side = 0; side < 2; ++side) {
    if (n[side] == 0) continue;
    const int grid = grid_for(n[side] * LANES, 256, 8);
    if (in[side]) {
      auto fn = h->bf16 ? cf_encode_kernel<LANES, true> : cf_encode_kernel<LANES, false>;
      fn<<<grid, 256, 0, s>>>(in[side], n[side], st[side]);
    }
    if (out[side]) {
      auto fn = h->bf16 ? cf_decode_kernel<LANES, true> : cf_decode_kernel<LANES, false>;
      fn<<<grid, 256, 0, s>>>(st[side], n[side], out[side]);
    }
    CG_LAUNCH_CHECK();
  }
  return CG_OK;
}

int codec_dispatch(cg_bipartite* h, const float* P, const float* Q, float* Pout, float* Qout,
                   cudaStream_t s) {
  switch (h->K) {
    case 16: return codec<2>(h, P, Q, Pout, Qout, s);
    case 32: return codec<4>(h, P, Q, Pout, Qout, s);
    default: return codec<8>(h, P, Q, Pout, Qout, s);
  }
}

void cf_free(cg_bipartite* h) {
  for (int s = 0; s < 2; ++s) cf_pieces_free(&h->side[s]);  // with the lists
  cudaFree(h->P);  // with Q, the partials and the counter
  delete h;
}

// Lists the vertices with more than kCfWide pieces from the list's front and
// those with more than kCfWarp from its end (cap is at least the number of
// either together).  Each vertex's update is its own: the order is of no account.
__global__ void many_pieces_kernel(const int64_t* __restrict__ poff, int64_t n, int32_t cap,
                                   int32_t* __restrict__ list, int32_t* __restrict__ count) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int64_t np = poff[v + 1] - poff[v];
    if (np > kCfWide)
      list[atomicAdd(count, 1)] = (int32_t)v;
    else if (np > kCfWarp)
      list[cap - 1 - atomicAdd(count + 1, 1)] = (int32_t)v;
  }
}

int build_pieces(cg_bipartite* h, int side, cudaStream_t s) {
  const int64_t* off = side == 0 ? h->uoff : h->ioff;
  const int64_t n = side == 0 ? h->U : h->I;
  CG_TRY(cf_pieces_build(&h->side[side], n, h->R, h->K, off, kCfWarp, s));
  const CfPieces& c = h->side[side];
  h->bytes += c.bytes;
  // vertices with many pieces get a warp or a whole block in the update
  const int32_t cap = c.most_many;
  h->wide[side] = c.many;
  int32_t* count = c.many + cap;
  CG_CUDA(cudaMemsetAsync(count, 0, 2 * sizeof(int32_t), s));
  if (n > 0) {
    many_pieces_kernel<<<grid_for(n, 256), 256, 0, s>>>(c.poff, n, cap, h->wide[side],
                                                        count);
    CG_LAUNCH_CHECK();
  }
  int32_t got[2] = {0, 0};
  CG_CUDA(cudaMemcpyAsync(got, count, sizeof(got), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  h->nwide[side] = got[0];
  h->nwarp[side] = got[1];
  h->warp[side] = h->wide[side] + cap - got[1];
  return CG_OK;
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int cf_transpose(int64_t U, int64_t I, const int64_t* uoff, const int32_t* uitem,
                 const uint8_t* urate, int64_t* ioff, int32_t* iuser, uint8_t* irate,
                 cudaStream_t stream) {
  CG_ARG(U >= 0 && I >= 1 && I < (int64_t)1 << 31, "cf_transpose: need U >= 0, 1 <= I < 2^31");
  CG_ARG(uoff && ioff, "cf_transpose: null offsets");
  int64_t R = 0;
  CG_CUDA(cudaMemcpyAsync(&R, uoff + U, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  CG_CUDA(cudaStreamSynchronize(stream));
  CG_ARG(R >= 0 && R < 0x7FFFFFFFLL, "cf_transpose: rating count %lld out of range",
         (long long)R);
  CG_ARG(R == 0 || (uitem && urate && iuser && irate), "cf_transpose: null rating arrays");
  int64_t* cnt = nullptr;
  int32_t *user = nullptr, *idx = nullptr, *order = nullptr, *bad = nullptr;
  uint32_t *key = nullptr, *key2 = nullptr;
  const size_t Rm = (size_t)(R > 0 ? R : 1);
  cudaError_t e = cudaMallocAsync((void**)&cnt, sizeof(int64_t) * (size_t)I, stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&bad, sizeof(int32_t), stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&user, sizeof(int32_t) * Rm, stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&idx, sizeof(int32_t) * Rm, stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&order, sizeof(int32_t) * Rm, stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&key, sizeof(uint32_t) * Rm, stream);
  if (e == cudaSuccess) e = cudaMallocAsync((void**)&key2, sizeof(uint32_t) * Rm, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(cnt, 0, sizeof(int64_t) * (size_t)I, stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(bad, 0, sizeof(int32_t), stream);
  int st = CG_OK;
  if (e == cudaSuccess && R > 0) {
    item_hist_kernel<<<grid_for(R, 256), 256, 0, stream>>>(uitem, R, I, cnt, bad);
    e = cudaGetLastError();
  }
  int32_t hbad = 0;
  if (e == cudaSuccess) e = cudaMemcpyAsync(&hbad, bad, sizeof(int32_t), cudaMemcpyDeviceToHost,
                                            stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  if (e == cudaSuccess && hbad) {
    set_error("cf_transpose: an item index is outside [0, %lld)", (long long)I);
    st = CG_ERR_INVALID_ARG;
  }
  if (e == cudaSuccess && st == CG_OK) st = exclusive_scan_i64(cnt, ioff, I, stream);
  if (e == cudaSuccess && st == CG_OK && R > 0) {
    expand_users_kernel<<<grid_for(U * 32, 256), 256, 0, stream>>>(uoff, U, uitem, user, key,
                                                                    idx);
    e = cudaGetLastError();
    int bits = 1;
    while (bits < 31 && ((int64_t)1 << bits) < I) ++bits;
    // stable sort by item: users stay ascending within each item
    if (e == cudaSuccess) st = radix_sort_pairs(key, idx, key2, order, R, bits, stream);
    if (e == cudaSuccess && st == CG_OK) {
      transpose_gather_kernel<<<grid_for(R, 256), 256, 0, stream>>>(order, R, user, urate, iuser,
                                                                    irate);
      e = cudaGetLastError();
    }
  }
  cudaFreeAsync(cnt, stream);
  cudaFreeAsync(bad, stream);
  cudaFreeAsync(user, stream);
  cudaFreeAsync(idx, stream);
  cudaFreeAsync(order, stream);
  cudaFreeAsync(key, stream);
  cudaFreeAsync(key2, stream);
  if (e != cudaSuccess) return cuda_fail(e, "cf_transpose", __FILE__, __LINE__);
  return st;
}

int cf_create(int64_t U, int64_t I, int32_t K, int32_t precision, const int64_t* uoff,
              const int32_t* uitem, const uint8_t* urate, const int64_t* ioff,
              const int32_t* iuser, const uint8_t* irate, cg_bipartite** out,
              cudaStream_t stream) {
  CG_ARG(out != nullptr, "cf_create: out is NULL");
  *out = nullptr;
  CG_ARG(U >= 1 && I >= 1 && U < (int64_t)1 << 31 && I < (int64_t)1 << 31,
         "cf_create: need 1 <= U, I < 2^31");
  CG_ARG(K == 16 || K == 32 || K == 64, "cf_create: K must be 16, 32 or 64 (got %d)", K);
  CG_ARG(precision >= 0 && precision <= 2,
         "cf_create: precision must be 0 (FP32), 1 (BF16) or 2 (BF16 hi+lo), got %d", precision);
  CG_ARG(uoff && ioff, "cf_create: null offsets");
  int64_t R = 0, R2 = 0;
  CG_CUDA(cudaMemcpyAsync(&R, uoff + U, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  CG_CUDA(cudaMemcpyAsync(&R2, ioff + I, sizeof(int64_t), cudaMemcpyDeviceToHost, stream));
  CG_CUDA(cudaStreamSynchronize(stream));
  CG_ARG(R == R2 && R >= 0, "cf_create: user side has %lld ratings, item side %lld",
         (long long)R, (long long)R2);
  CG_ARG(R == 0 || (uitem && urate && iuser && irate), "cf_create: null rating arrays");
  cg_bipartite* h = new cg_bipartite();
  CG_CUDA(cudaGetDevice(&h->device));
  h->U = U;
  h->I = I;
  h->R = R;
  h->K = K;
  h->bf16 = precision == 1;
  h->uoff = uoff;
  h->uitem = uitem;
  h->urate = urate;
  h->ioff = ioff;
  h->iuser = iuser;
  h->irate = irate;
  int st = build_pieces(h, 0, stream);
  if (st == CG_OK) st = build_pieces(h, 1, stream);
  cudaError_t e = cudaSuccess;
  const size_t el = h->bf16 ? 2 : 4;
  if (st == CG_OK) {
    st = cf_rows_grid(K, &h->gather_grid);
    const size_t pb = Scratch::round(el * (size_t)U * K), qb = Scratch::round(el * (size_t)I * K),
                 sb = Scratch::round(sizeof(double) * h->gather_grid);
    char* slab = nullptr;
    e = cudaMalloc((void**)&slab, pb + qb + sb + sizeof(unsigned));
    if (e == cudaSuccess) {
      h->P = slab;
      h->Q = slab + pb;
      h->partials = reinterpret_cast<double*>(slab + pb + qb);
      h->counter = reinterpret_cast<unsigned*>(slab + pb + qb + sb);
      h->bytes += (int64_t)(el * (size_t)(U + I) * K);
      e = cudaMemsetAsync(h->counter, 0, sizeof(unsigned), stream);
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(stream);
  }
  if (st == CG_OK && e != cudaSuccess) st = cuda_fail(e, "cf_create", __FILE__, __LINE__);
  if (st != CG_OK) {
    cudaStreamSynchronize(stream);
    cf_free(h);
    return st;
  }
  *out = h;
  return CG_OK;
}

int cf_destroy(cg_bipartite* h) {
  if (!h) return CG_OK;
  cudaDeviceSynchronize();
  cf_free(h);
  return CG_OK;
}

int cf_set_factors(cg_bipartite* h, const float* P, const float* Q, cudaStream_t stream) {
  CG_ARG(h && P && Q, "cf_set_factors: null argument");
  return codec_dispatch(h, P, Q, nullptr, nullptr, stream);
}

int cf_get_factors(const cg_bipartite* h, float* P, float* Q, cudaStream_t stream) {
  CG_ARG(h, "cf_get_factors: null handle");
  return codec_dispatch(const_cast<cg_bipartite*>(h), nullptr, nullptr, P, Q, stream);
}

int cf_sweep(cg_bipartite* h, int32_t sweeps, double lambda, double step, double* sse,
             cudaStream_t stream) {
  CG_ARG(h, "cf_sweep: null handle");
  CG_ARG(sweeps >= 1, "cf_sweep: sweeps must be >= 1");
  CG_ARG(lambda >= 0.0 && step >= 0.0, "cf_sweep: lambda and step must be >= 0");
  for (int t = 0; t < sweeps; ++t)
    for (int phase = 0; phase < 4; ++phase)
      CG_TRY(run_phase(h, phase, sse ? sse + t : nullptr, (float)lambda, (float)step, stream));
  return CG_OK;
}

int cf_sweep_phase(cg_bipartite* h, int32_t phase, double lambda, double step, double* sse,
                   cudaStream_t stream) {
  CG_ARG(h, "cf_sweep_phase: null handle");
  CG_ARG(phase >= 0 && phase <= 3, "cf_sweep_phase: phase must be in [0, 3]");
  return run_phase(h, phase, sse, (float)lambda, (float)step, stream);
}

int cf_info(const cg_bipartite* h, int64_t* ratings, int64_t* user_pieces, int64_t* item_pieces,
            int64_t* bytes) {
  CG_ARG(h, "cf_info: null handle");
  if (ratings) *ratings = h->R;
  if (user_pieces) *user_pieces = h->side[0].npieces;
  if (item_pieces) *item_pieces = h->side[1].npieces;
  if (bytes) *bytes = h->bytes;
  return CG_OK;
}

}  // extern "C"
