// Building the staged segments' stream (staged_stream.cuh): rows sorted by
// (window, length class), cut into tasks, indices and row positions laid out
// task by task.
#include <algorithm>

#include "staged_stream.cuh"

namespace cg {
namespace {

constexpr int kClassSpace = 1 << kClassBits;

__device__ __forceinline__ int last_le64(const int64_t* a, int n, int64_t v) {
  int lo = 0, hi = n;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (a[mid] <= v) lo = mid + 1; else hi = mid;
  }
  return lo - 1;
}

// Sort key of every row: its window and the class of its last 1..kStagedMost
// edges; nfull: its full pieces (their total in *total).
__global__ void staged_key_kernel(const int32_t* __restrict__ rp, int64_t rows,
                                  const int64_t* __restrict__ row_base,
                                  const int64_t* __restrict__ wbase, int m2,
                                  uint32_t* __restrict__ key, int32_t* __restrict__ val,
                                  int32_t* __restrict__ nfull,
                                  unsigned long long* __restrict__ total) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x) {
    const int s = last_le64(row_base, m2, r);
    const int len = rp[r + 1] - rp[r];
    const int full = (len - 1) / kStagedMost;
    const uint32_t win = (uint32_t)(wbase[s] + (r - row_base[s]) / kStagedWindow);
    key[r] = (win << kClassBits) | (uint32_t)staged_class(len - full * kStagedMost);
    val[r] = (int32_t)r;
    nfull[r] = full;
    if (full) atomicAdd(total, (unsigned long long)full);
  }
}

// The full pieces: piece j of row r is item rows + pos[r] + j.
__global__ void staged_extra_kernel(const int32_t* __restrict__ nfull,
                                    const int64_t* __restrict__ pos, int64_t rows,
                                    uint32_t* __restrict__ key, int32_t* __restrict__ val,
                                    int32_t* __restrict__ xrow, int32_t* __restrict__ xpiece) {
  for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < rows;
       r += (int64_t)gridDim.x * blockDim.x)
    for (int j = 0; j < nfull[r]; ++j) {
      const int64_t x = pos[r] + j;
      key[rows + x] = (key[r] & ~(uint32_t)(kClassSpace - 1)) | kClassFull;
      val[rows + x] = (int32_t)(rows + x);
      xrow[x] = (int32_t)r;
      xpiece[x] = j;
    }
}

// Per bucket (window, class): its first sorted item, its tasks and their size
// in 32-byte units.
__global__ void staged_bucket_kernel(const uint32_t* __restrict__ skey, int64_t n, int64_t nb,
                                     int64_t* __restrict__ start, int32_t* __restrict__ tasks,
                                     int32_t* __restrict__ units) {
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b <= nb;
       b += (int64_t)gridDim.x * blockDim.x) {
    int64_t at[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      int64_t lo = h ? at[0] : 0, hi = n;
      while (lo < hi) {
        const int64_t mid = (lo + hi) >> 1;
        if ((int64_t)skey[mid] < b + h) lo = mid + 1; else hi = mid;
      }
      at[h] = lo;
    }
    start[b] = at[0];
    if (b == nb) break;
    const int c = (int)(b & (kClassSpace - 1));
    int t = 0, u = 0;
    if (c <= kClassFull) {
      t = (int)((at[1] - at[0] + class_rows(c) - 1) / class_rows(c));
      u = t * class_units(c);
    }
    tasks[b] = t;
    units[b] = u;
  }
}

// First task of each segment.
__global__ void staged_seg_task_kernel(const int64_t* __restrict__ task_base,
                                       const int64_t* __restrict__ wbase, int m2, int k,
                                       int32_t* __restrict__ seg_task) {
  for (int q = blockIdx.x * blockDim.x + threadIdx.x; q <= k; q += gridDim.x * blockDim.x)
    seg_task[q] = (int32_t)task_base[wbase[q < m2 ? q : m2] << kClassBits];
}

// One warp per task: its descriptor, its index words and its rows' positions.
__global__ void __launch_bounds__(256)
staged_fill_kernel(const uint32_t* __restrict__ colf, const int32_t* __restrict__ rp,
                   const int64_t* __restrict__ row_base, const int64_t* __restrict__ edge_base,
                   const int64_t* __restrict__ cstart, const int64_t* __restrict__ wbase, int m2,
                   const int32_t* __restrict__ item, int64_t rows,
                   const int32_t* __restrict__ xrow, const int32_t* __restrict__ xpiece,
                   const int64_t* __restrict__ start, const int64_t* __restrict__ task_base,
                   const int64_t* __restrict__ unit_base, int nb, int64_t ntasks, int pad,
                   int64_t carry_base, const int32_t* __restrict__ place,
                   uint4* __restrict__ desc, uint8_t* __restrict__ cs) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < ntasks; t += nw) {
    const int b = last_le64(task_base, nb, t);
    const int c = b & (kClassSpace - 1);
    const int64_t win = b >> kClassBits;
    const int s = last_le64(wbase, m2, win);
    const int64_t off = unit_base[b] + (t - task_base[b]) * class_units(c);
    const int64_t first = start[b] + (t - task_base[b]) * class_rows(c);
    const int n = (int)min((int64_t)class_rows(c), start[b + 1] - first);
    const int64_t row0 = row_base[s] + (win - wbase[s]) * kStagedWindow;
    const int64_t shift = cstart[s] - edge_base[s];
    const int words = class_words(c), slots = class_slots(c), lg = class_lg(c);
    uint8_t* base = cs + off * 32;
    if (lane == 0) {
      const int64_t z =
          c == kClassFull ? carry_base + (item[first] - rows) : place ? 0 : row0;
      desc[t] = make_uint4((uint32_t)off, class_word(c), (uint32_t)z, 0u);
    }
    // edges [e0, e0 + len) of the row slot j of the task (len 0: unused)
    auto row_of = [&](int j, int64_t* e0, int* len) -> int32_t {
      *len = 0;
      *e0 = 0;
      if (j >= n) return -1;
      const int32_t it = item[first + j];
      const int64_t r = it < rows ? it : xrow[it - rows];
      const int whole = rp[r + 1] - rp[r];
      const int full = (whole - 1) / kStagedMost;
      const int piece = it < rows ? full : xpiece[it - rows];
      *e0 = (int64_t)rp[r] + (int64_t)piece * kStagedMost;
      *len = it < rows ? whole - full * kStagedMost : kStagedMost;
      return place ? place[r] : (int32_t)(r - row0);
    };
    auto put = [&](int slot, uint32_t v) {
      reinterpret_cast<uint16_t*>(base)[2 * word_at(words, slot >> 1, lane) + (slot & 1)] =
          (uint16_t)v;
    };
    if (c < 8) {
      const int R = short_rows(c), L = c + 1;
      const int np = class_pos(c);
      uint16_t* pos = reinterpret_cast<uint16_t*>(base + words * 128) + lane * 2 * np;
      for (int q = 0; q < R; ++q) {
        int64_t e0;
        int len;
        const int32_t id = row_of(q * 32 + lane, &e0, &len);
        for (int l = 0; l < L; ++l)
          put(q * L + l, l < len ? colf[e0 + l + shift] & 0xFFFFu : (uint32_t)pad);
        pos[q] = (uint16_t)(id < 0 ? kNoRow : (uint32_t)id);
      }
      for (int q = R; q < 2 * np; ++q) pos[q] = (uint16_t)kNoRow;
    } else {
      int64_t e0;
      int len;
      const int j = lane >> lg, sub = lane & ((1 << lg) - 1);
      const int32_t id = row_of(j, &e0, &len);
      for (int i = 0; i < slots; ++i) {
        const int e = (i << lg) + sub;
        put(i, e < len ? colf[e0 + e + shift] & 0xFFFFu : (uint32_t)pad);
      }
      if (sub == 0)
        reinterpret_cast<uint16_t*>(base + words * 128)[j] =
            (uint16_t)(id < 0 ? kNoRow : c == kClassFull ? 0u : (uint32_t)id);
    }
    for (int i = slots; i < 2 * words; ++i) put(i, (uint32_t)pad);
  }
}

}  // namespace

int staged_build(SegPlan* p, int m2, int pad, int64_t carry_base, cudaStream_t s,
                 const int32_t* place) {
  const int k = p->k;
  const int64_t rows = p->row_base[m2];
  p->h_seg_task.assign(k + 1, 0);
  if (rows == 0) {
    CG_CUDA(cudaMemsetAsync(p->seg_task, 0, sizeof(int32_t) * (size_t)(k + 1), s));
    return seg_plan_carries(p, carry_base);
  }
  std::vector<int64_t> wbase(m2 + 1, 0);
  for (int q = 0; q < m2; ++q)
    wbase[q + 1] = wbase[q] + ceil_div(p->row_base[q + 1] - p->row_base[q], kStagedWindow);
  const int64_t nb = wbase[m2] << kClassBits;
  if (nb >= 0x7FFFFFFFLL) {
    set_error("staged segments: too many of them (%d)", m2);
    return CG_ERR_UNSUPPORTED;
  }
  const int64_t edges = p->edge_base[m2];
  const int64_t most = rows + edges / kStagedMost;  // rows and at most their full pieces
  Scratch tmp(s, p->lent, p->lent_bytes,
              6 * Scratch::round(4 * (size_t)most) + sort_scratch(most) +
                  3 * Scratch::round(8 * (size_t)(nb + 1)) + 2 * Scratch::round(4 * (size_t)nb) +
                  2 * scan_scratch(nb) + Scratch::round(8 * (size_t)(rows + 1)) +
                  scan_scratch(rows) + Scratch::round(8 * (size_t)(m2 + 1)) + 4096);
  int64_t *d_wbase = nullptr, *pos = nullptr, *start = nullptr, *task_base = nullptr,
          *unit_base = nullptr;
  uint32_t *key = nullptr, *skey = nullptr;
  int32_t *val = nullptr, *item = nullptr, *nfull = nullptr, *tasks = nullptr, *units = nullptr,
          *xrow = nullptr, *xpiece = nullptr;
  unsigned long long* total = nullptr;
  CG_CUDA(tmp.get(&d_wbase, m2 + 1));
  CG_CUDA(tmp.get(&total, 1));
  CG_CUDA(tmp.get(&nfull, rows));
  CG_CUDA(cudaMemcpyAsync(d_wbase, wbase.data(), sizeof(int64_t) * (m2 + 1),
                          cudaMemcpyHostToDevice, s));
  CG_CUDA(cudaMemsetAsync(total, 0, sizeof(unsigned long long), s));
  CG_CUDA(tmp.get(&key, most));
  CG_CUDA(tmp.get(&skey, most));
  CG_CUDA(tmp.get(&val, most));
  CG_CUDA(tmp.get(&item, most));
  staged_key_kernel<<<grid_for(rows, 256), 256, 0, s>>>(p->rp32, rows, p->meta, d_wbase, m2, key,
                                                        val, nfull, total);
  CG_LAUNCH_CHECK();
  unsigned long long nx = 0;
  CG_CUDA(cudaMemcpyAsync(&nx, total, sizeof(nx), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  CG_TRY(seg_plan_carries(p, carry_base + (int64_t)nx));
  xrow = p->carry_row + carry_base;
  CG_CUDA(tmp.get(&xpiece, nx));
  if (nx > 0) {
    CG_CUDA(tmp.get(&pos, rows + 1));
    CG_TRY(exclusive_scan_i32_to_i64(nfull, pos, rows, s, &tmp));
    staged_extra_kernel<<<grid_for(rows, 256), 256, 0, s>>>(nfull, pos, rows, key, val, xrow,
                                                            xpiece);
    CG_LAUNCH_CHECK();
  }
  const int64_t n = rows + (int64_t)nx;
  int bits = kClassBits;
  while (bits < 32 && ((int64_t)1 << bits) < nb) ++bits;
  CG_TRY(radix_sort_pairs(key, val, skey, item, n, bits, s, &tmp));
  CG_CUDA(tmp.get(&start, nb + 1));
  CG_CUDA(tmp.get(&tasks, nb));
  CG_CUDA(tmp.get(&units, nb));
  CG_CUDA(tmp.get(&task_base, nb + 1));
  CG_CUDA(tmp.get(&unit_base, nb + 1));
  staged_bucket_kernel<<<grid_for(nb + 1, 256), 256, 0, s>>>(skey, n, nb, start, tasks, units);
  CG_LAUNCH_CHECK();
  CG_TRY(exclusive_scan_i32_to_i64(tasks, task_base, nb, s, &tmp));
  CG_TRY(exclusive_scan_i32_to_i64(units, unit_base, nb, s, &tmp));
  staged_seg_task_kernel<<<grid_for(k + 1, 128), 128, 0, s>>>(task_base, d_wbase, m2, k,
                                                              p->seg_task);
  CG_LAUNCH_CHECK();
  int64_t nunits = 0;
  CG_CUDA(cudaMemcpyAsync(&nunits, unit_base + nb, sizeof(int64_t), cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaMemcpyAsync(p->h_seg_task.data(), p->seg_task, sizeof(int32_t) * (k + 1),
                          cudaMemcpyDeviceToHost, s));
  CG_CUDA(cudaStreamSynchronize(s));
  const int64_t ntasks = p->h_seg_task[k];
  // descriptors and stream, one allocation (desc owns it); the prefetch reads ahead
  const int64_t db = (int64_t)Scratch::round(sizeof(uint4) * (size_t)ntasks);
  const int64_t bytes = db + nunits * 32 + 2 * kStreamAhead;
  if (bytes > p->cs_cap) {
    cudaFree(p->desc);
    p->desc = nullptr;
    p->cs_cap = 0;
    CG_CUDA(cudaMalloc((void**)&p->desc, (size_t)bytes));
    p->cs_cap = bytes;
  }
  p->cs = reinterpret_cast<uint8_t*>(p->desc) + db;
  staged_fill_kernel<<<grid_for(ntasks * 32, 256), 256, 0, s>>>(
      p->colf, p->rp32, p->meta, p->meta + (k + 1), p->meta + 2 * (k + 1), d_wbase, m2, item,
      rows, xrow, xpiece, start, task_base, unit_base, (int)nb, ntasks, pad, carry_base, place,
      p->desc, p->cs);
  CG_LAUNCH_CHECK();
  return CG_OK;
}

}  // namespace cg
