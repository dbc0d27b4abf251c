// Label propagation over the segmented graph (the paper's LP application,
// Table IV): synchronous passes L'[v] = min(L[v], min over in-neighbours u of
// L[u]) -- Algorithm 3's gather with a min, Algorithm 4's merge with a min,
// fused with the label update and a count of changed labels.  Integer
// arithmetic throughout: results are exact.
#include "handles.cuh"
#include "update.cuh"

namespace cg {
namespace {

// Merge of one warp-owned block with the min operator (same walk as the
// PageRank merge), then L' = min(L, acc) and the number of changed labels, added
// to *changed.  With a pin, the last block to finish (done) writes the sum and
// the ticket there and clears both counters for the next pass.
__global__ void __launch_bounds__(kMergeWarps * 32)
lp_merge_update_kernel(const int32_t* blk, const int32_t* idx_map,
                       const int32_t* interm, int k, int nb, int B, int32_t V,
                       const int32_t* labels_in, int32_t* labels_out,
                       unsigned long long* changed, unsigned* done,
                       volatile unsigned long long* pin, unsigned long long ticket) {
  extern __shared__ int32_t lp_acc_all[];
  if (!chain_begin()) return;
  const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t mb = (int64_t)blockIdx.x * kMergeWarps + w;
  unsigned long long cnt = 0;
  if (mb < nb) {
    int32_t* acc = lp_acc_all + (int64_t)w * B;
    const int64_t v0 = mb * B;
    const int n = (int)((V - v0) < B ? (V - v0) : B);
    warp_merge<MinI32>(blk, idx_map, interm, k, nb, mb, v0, n, acc);
    constexpr int U = 4;  // labels per lane loaded together
    for (int i0 = lane; i0 < n; i0 += 32 * U) {
      int32_t old[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        old[u] = i0 + 32 * u < n ? __ldcs(labels_in + v0 + i0 + 32 * u) : 0;
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + 32 * u;
        if (i < n) {
          const int32_t l = acc[i] < old[u] ? acc[i] : old[u];
          __stcs(labels_out + v0 + i, l);
          cnt += (l != old[u]);
        }
      }
    }
  }
  cnt = warp_sum(cnt);
  if (!pin) {
    if (lane == 0 && cnt) atomicAdd(changed, cnt);
    return;
  }
  __shared__ unsigned s_cnt;
  if (threadIdx.x == 0) s_cnt = 0u;
  __syncthreads();
  if (lane == 0 && cnt) atomicAdd(&s_cnt, (unsigned)cnt);
  __syncthreads();
  if (threadIdx.x != 0) return;
  if (s_cnt) atomicAdd(changed, (unsigned long long)s_cnt);
  __threadfence();
  if (atomicAdd(done, 1u) != gridDim.x - 1) return;
  __threadfence();
  pin[0] = atomicExch(changed, 0ull);
  __threadfence_system();
  pin[1] = ticket;
  *done = 0u;
}

// One pass; with a pin the count goes there (see the kernel).
int lp_pass(const cg_segmented* g, const int32_t* labels_in, int32_t* labels_out,
            unsigned long long* cnt, unsigned long long* pin, unsigned long long ticket,
            cudaStream_t stream) {
  CG_TRY(run_seg_gather<MinI32>(g->plan, labels_in, g->V, (int32_t*)g->interm, stream));
  const size_t smem = (size_t)kMergeWarps * g->mB * 4;
  if (smem > 32 * 1024)
    CG_CUDA(cudaFuncSetAttribute((const void*)lp_merge_update_kernel,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  return launch_chained(lp_merge_update_kernel, (unsigned)ceil_div(g->mnb, kMergeWarps),
                        kMergeWarps * 32, smem, stream, g->blk, g->idx_map,
                        (const int32_t*)g->interm, g->k, g->mnb, g->mB, g->V, labels_in,
                        labels_out, cnt, g->counter, pin, ticket);
}

}  // namespace
}  // namespace cg

using namespace cg;

extern "C" {

int lp_iterate(const cg_segmented* g, const int32_t* labels_in, int32_t* labels_out,
               int64_t* dev_changed, int64_t* host_changed, cudaStream_t stream) {
  CG_ARG(g && labels_in && labels_out, "lp_iterate: null argument");
  CG_ARG(labels_in != labels_out, "lp_iterate: labels_out must not alias labels_in");
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(dev_changed);
  if (!cnt) cnt = reinterpret_cast<unsigned long long*>(g->dslot + 3);
  CG_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), stream));
  CG_TRY(lp_pass(g, labels_in, labels_out, cnt, nullptr, 0, stream));
  if (host_changed) {
    unsigned long long h = 0;
    CG_CUDA(cudaMemcpyAsync(&h, cnt, sizeof(h), cudaMemcpyDeviceToHost, stream));
    CG_CUDA(cudaStreamSynchronize(stream));
    *host_changed = (int64_t)h;
  }
  return CG_OK;
}

int lp_run(const cg_segmented* g, int32_t* labels, int64_t max_passes, int64_t* host_passes,
           int64_t* host_changes, cudaStream_t stream) {
  CG_ARG(g && labels && host_passes, "lp_run: null argument");
  CG_ARG(max_passes >= 1, "lp_run: max_passes must be >= 1");
  int32_t* a = labels;
  int32_t* b = reinterpret_cast<int32_t*>(g->rank_tmp);  // V int32 of handle scratch
  if (!g->pin) {
    CG_CUDA(cudaHostAlloc((void**)&g->pin, 2 * sizeof(unsigned long long), 0));
    g->pin[0] = g->pin[1] = 0;
  }
  unsigned long long* cnt = reinterpret_cast<unsigned long long*>(g->dslot + 3);
  CG_CUDA(cudaMemsetAsync(cnt, 0, sizeof(unsigned long long), stream));
  int64_t p = 0;
  for (; p < max_passes;) {
    CG_TRY(lp_pass(g, a, b, cnt, g->pin, ++g->ticket, stream));
    CG_TRY(wait_ticket(g->pin + 1, g->ticket, stream, "lp_run"));
    const int64_t changed = (int64_t)g->pin[0];
    if (host_changes) host_changes[p] = changed;
    ++p;
    int32_t* t = a;
    a = b;
    b = t;
    if (changed == 0) break;
  }
  if (a != labels)
    CG_CUDA(cudaMemcpyAsync(labels, a, sizeof(int32_t) * (size_t)g->V, cudaMemcpyDeviceToDevice,
                            stream));
  CG_CUDA(cudaStreamSynchronize(stream));
  *host_passes = p;
  return CG_OK;
}

}  // extern "C"
