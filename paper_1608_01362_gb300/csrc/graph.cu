// Degrees, frequency-based clustering and CSR renumbering (Section V).
#include "rowwalk.cuh"

namespace cg {
namespace {

// Out-degree by counting sources, one reduction per edge: bound by the L2's
// atomics.  A warp combines the equal ones of 32 edges first (match_any) while it
// meets any: it looks at the first of every four batches, and combines the
// batches of four looks in a row from one that had equal sources on.  65 M edges:
// RMAT 382 us (511 combining always, 378 never), one source in every edge 1337
// (1337, 41,760), in every 16th 1645 (1653, 2846), sources V x^6 3694 (3680, 5758).
__global__ void __launch_bounds__(256)
out_degree_kernel(const int32_t* __restrict__ src, int64_t E, int32_t V,
                  int32_t* __restrict__ outdeg) {
  constexpr int U = 4, kLooks = 4;
  constexpr unsigned kFull = 0xffffffffu;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int lane = threadIdx.x & 31;
  int left = 0;  // looks whose batches are still combined
  // (base is that of lane 0: the warp stays together)
  for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); base < E;
       base += stride * U) {
    int32_t u[U];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int64_t e = base + lane + j * stride;
      u[j] = e < E ? __ldcs(src + e) : -1;
      if (u[j] >= V) u[j] = -1;  // out of range: ignored
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (j == 0 || left > 0) {
        const unsigned peers =
            __match_any_sync(kFull, u[j] >= 0 ? (unsigned)u[j] : (0x80000000u | (unsigned)lane));
        if (j == 0) left = __any_sync(kFull, peers & (peers - 1)) ? kLooks : max(left - 1, 0);
        if (u[j] >= 0 && lane == __ffs(peers) - 1) atomicAdd(outdeg + u[j], __popc(peers));
      } else if (u[j] >= 0) {
        atomicAdd(outdeg + u[j], 1);
      }
    }
  }
}

__global__ void inv_outdeg_kernel(const int32_t* __restrict__ outdeg, int32_t V,
                                  float* __restrict__ inv) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    const int32_t d = outdeg[v];
    inv[v] = d > 0 ? 1.0f / (float)d : 0.0f;
  }
}

// Sort key: hotter (larger degree key) first -> ascending (INT32_MAX - key).
__global__ void cluster_key_kernel(const int32_t* __restrict__ outdeg, int32_t V, int32_t thr,
                                   uint32_t* __restrict__ key, int32_t* __restrict__ val) {
  for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < V;
       v += (int64_t)gridDim.x * blockDim.x) {
    int32_t d = outdeg[v];
    if (d < 0) d = 0;
    key[v] = (uint32_t)(0x7FFFFFFF - d / thr);
    val[v] = (int32_t)v;
  }
}

__global__ void invert_perm_kernel(const int32_t* __restrict__ old_of_new, int32_t V,
                                   int32_t* __restrict__ new_of_old) {
  for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < V;
       n += (int64_t)gridDim.x * blockDim.x)
    new_of_old[old_of_new[n]] = (int32_t)n;
}

__global__ void relabel_len_kernel(const int64_t* __restrict__ offsets,
                                   const int32_t* __restrict__ old_of_new, int32_t V,
                                   int64_t* __restrict__ len) {
  for (int64_t n = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; n < V;
       n += (int64_t)gridDim.x * blockDim.x) {
    const int64_t o = old_of_new[n];
    len[n] = (o >= 0 && o < V) ? offsets[o + 1] - offsets[o] : 0;
  }
}

// The new rows' sources, mapped to new IDs: a warp takes kRelabelTile
// consecutive edges of the new CSR, finds each edge's new row (rowwalk.cuh),
// and reads its source at the same place of the old row.  Bound by the random
// 4-byte reads of new_of_old (L2 sectors).  65.2 M edges: 2.49 ms with a warp
// per row (15 edges a row, most lanes idle) -> 0.43 ms.
// (PosT: int64 where there are 2^31 edges and more.)
constexpr int kRelabelTile = 1024;

template <typename PosT>
__global__ void __launch_bounds__(256)
relabel_copy_kernel(const int64_t* __restrict__ offsets, const int32_t* __restrict__ src,
                    const int32_t* __restrict__ new_of_old,
                    const int32_t* __restrict__ old_of_new, int32_t V, int64_t E,
                    const int64_t* __restrict__ out_offsets, int32_t* __restrict__ out_src) {
  constexpr int U = 4;  // batches of 32 edges whose reads are in flight together
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t n = min(E, out_offsets[V]);  // an old_of_new that is no permutation
  RowWalk<int64_t, PosT> walk(out_offsets, V, (PosT)n);
  for (int64_t b = ((((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5)) * kRelabelTile; b < n;
       b += nw * kRelabelTile) {
    walk.seek((PosT)b);
    for (int i = 0; i < kRelabelTile && b + i < n; i += 32 * U) {
      int64_t at[U];
      int32_t u[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int64_t e = b + i + 32 * j + lane;
        PosT st, en;
        const int32_t r = walk.row_of((PosT)e, e < n, &st, &en);
        at[j] = -1;
        if (e < n) {
          const int64_t o = __ldg(old_of_new + r);  // in [0, V): its row is not empty
          at[j] = __ldg(offsets + o) + (e - st);
        }
      }
#pragma unroll
      for (int j = 0; j < U; ++j) u[j] = at[j] >= 0 ? __ldcs(src + at[j]) : -1;
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const int32_t m = (u[j] >= 0 && u[j] < V) ? __ldg(new_of_old + u[j]) : u[j];
        if (at[j] >= 0) __stcs(out_src + b + i + 32 * j + lane, m);
      }
    }
  }
}

// Rows of w 16-byte words: out[i] = in[idx[i]] (zeros where idx[i] is out of range).
__global__ void permute_rows_kernel(const uint4* __restrict__ in, const int32_t* __restrict__ idx,
                                    int64_t n, int64_t n_in, int w, uint4* __restrict__ out) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < n * w;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = t / w, c = t - i * w;
    const int32_t j = idx[i];
    out[t] = (j >= 0 && j < n_in) ? in[(int64_t)j * w + c] : make_uint4(0u, 0u, 0u, 0u);
  }
}

template <typename W>
__global__ void permute_kernel(const W* __restrict__ in, const int32_t* __restrict__ idx,
                               int64_t n, int64_t n_in, W* __restrict__ out) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t j = idx[i];
    out[i] = (j >= 0 && j < n_in) ? in[j] : W(0);
  }
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int cg_out_degree(const int32_t* src, int64_t E, int32_t V, int32_t* outdeg,
                  cudaStream_t stream) {
  CG_ARG(V >= 1, "cg_out_degree: V must be >= 1 (got %d)", V);
  CG_ARG(E >= 0, "cg_out_degree: E must be >= 0");
  CG_ARG(outdeg && (E == 0 || src), "cg_out_degree: null pointer");
  CG_CUDA(cudaMemsetAsync(outdeg, 0, sizeof(int32_t) * (size_t)V, stream));
  if (E == 0) return CG_OK;
  out_degree_kernel<<<grid_for(E, 256), 256, 0, stream>>>(src, E, V, outdeg);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_inv_outdeg(const int32_t* outdeg, int32_t V, float* inv, cudaStream_t stream) {
  CG_ARG(V >= 1 && outdeg && inv, "cg_inv_outdeg: bad arguments");
  inv_outdeg_kernel<<<grid_for(V, 256), 256, 0, stream>>>(outdeg, V, inv);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_cluster(const int32_t* outdeg, int32_t V, int64_t E, int32_t mode, int32_t* new_of_old,
               int32_t* old_of_new, cudaStream_t stream) {
  CG_ARG(V >= 1 && E >= 0, "cg_cluster: V must be >= 1 and E >= 0");
  CG_ARG(outdeg && new_of_old && old_of_new, "cg_cluster: null pointer");
  CG_ARG(mode == 0 || mode == 1, "cg_cluster: mode must be 0 or 1 (got %d)", mode);
  CG_ARG(new_of_old != old_of_new, "cg_cluster: outputs must not alias");
  int64_t thr = 1;
  if (mode == 1) {
    thr = E / V;
    if (thr < 1) thr = 1;
    if (thr > 0x7FFFFFFF) thr = 0x7FFFFFFF;
  }
  Scratch tmp(stream, 3 * Scratch::round(4 * (size_t)V) + sort_scratch(V));
  uint32_t* key = nullptr;
  uint32_t* key2 = nullptr;
  int32_t* val = nullptr;
  CG_CUDA(tmp.get(&key, V));
  CG_CUDA(tmp.get(&key2, V));
  CG_CUDA(tmp.get(&val, V));
  cluster_key_kernel<<<grid_for(V, 256), 256, 0, stream>>>(outdeg, V, (int32_t)thr, key, val);
  CG_LAUNCH_CHECK();
  CG_TRY(radix_sort_pairs(key, val, key2, old_of_new, V, 31, stream, &tmp));
  invert_perm_kernel<<<grid_for(V, 256), 256, 0, stream>>>(old_of_new, V, new_of_old);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_permute4(const void* in, int64_t n_in, const int32_t* idx, int64_t n, void* out,
                cudaStream_t stream) {
  CG_ARG(n >= 0 && n_in >= 0, "cg_permute4: negative size");
  if (n == 0) return CG_OK;
  CG_ARG(in && idx && out && in != out, "cg_permute4: null or aliased pointer");
  permute_kernel<uint32_t><<<grid_for(n, 256), 256, 0, stream>>>((const uint32_t*)in, idx, n,
                                                                 n_in, (uint32_t*)out);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_permute8(const void* in, int64_t n_in, const int32_t* idx, int64_t n, void* out,
                cudaStream_t stream) {
  CG_ARG(n >= 0 && n_in >= 0, "cg_permute8: negative size");
  if (n == 0) return CG_OK;
  CG_ARG(in && idx && out && in != out, "cg_permute8: null or aliased pointer");
  CG_ARG(((uintptr_t)in & 7) == 0 && ((uintptr_t)out & 7) == 0,
         "cg_permute8: buffers must be 8-byte aligned");
  permute_kernel<uint64_t><<<grid_for(n, 256), 256, 0, stream>>>((const uint64_t*)in, idx, n,
                                                                 n_in, (uint64_t*)out);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_permute_rows(const void* in, int64_t n_in, int32_t row_bytes, const int32_t* idx,
                    int64_t n, void* out, cudaStream_t stream) {
  CG_ARG(n >= 0 && n_in >= 0, "cg_permute_rows: negative size");
  CG_ARG(row_bytes > 0 && row_bytes % 16 == 0, "cg_permute_rows: row_bytes must be a positive "
         "multiple of 16 (got %d)", row_bytes);
  if (n == 0) return CG_OK;
  CG_ARG(in && idx && out && in != out, "cg_permute_rows: null or aliased pointer");
  CG_ARG(((uintptr_t)in | (uintptr_t)out) % 16 == 0, "cg_permute_rows: rows need 16-byte "
         "aligned buffers");
  const int w = row_bytes / 16;
  permute_rows_kernel<<<grid_for(n * w, 256), 256, 0, stream>>>((const uint4*)in, idx, n, n_in, w,
                                                                (uint4*)out);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

int cg_relabel_csr(const int64_t* offsets, const int32_t* src, int32_t V, int64_t E,
                   const int32_t* new_of_old, const int32_t* old_of_new, int64_t* out_offsets,
                   int32_t* out_src, cudaStream_t stream) {
  CG_ARG(V >= 1 && E >= 0, "cg_relabel_csr: V must be >= 1 and E >= 0");
  CG_ARG(offsets && new_of_old && old_of_new && out_offsets && (E == 0 || (src && out_src)),
         "cg_relabel_csr: null pointer");
  CG_ARG((E == 0 || (const void*)out_src != (const void*)src) &&
             (const void*)out_offsets != (const void*)offsets,
         "cg_relabel_csr: outputs must not alias inputs");
  Scratch tmp(stream, Scratch::round(8 * ((size_t)V + 1)) + scan_scratch(V));
  int64_t* len = nullptr;
  CG_CUDA(tmp.get(&len, (size_t)V + 1));
  relabel_len_kernel<<<grid_for(V, 256), 256, 0, stream>>>(offsets, old_of_new, V, len);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i64(len, out_offsets, V, stream, &tmp));
  if (E > 0) {
    auto fn = E < 0x7FFFFFFFLL ? relabel_copy_kernel<int32_t> : relabel_copy_kernel<int64_t>;
    fn<<<grid_for(ceil_div(E, kRelabelTile) * 32, 256), 256, 0, stream>>>(
        offsets, src, new_of_old, old_of_new, V, E, out_offsets, out_src);
    CG_LAUNCH_CHECK();
  }
  return CG_OK;
}

}  // extern "C"
