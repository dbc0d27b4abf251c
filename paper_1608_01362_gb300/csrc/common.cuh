// Shared host/device helpers of the cagra_gb CUDA library: status codes,
// thread-local error text, device properties, block reductions.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>
#include <stdio.h>

#include <string>
#include <vector>

#include "../../include/cagra_gb.h"

namespace cg {

// Thread-local last error text (read through cg_last_error_message()).
void set_error(const char* fmt, ...);
const char* last_error();

// Record a CUDA error and return CG_ERR_CUDA (or CG_ERR_OOM).
int cuda_fail(cudaError_t e, const char* what, const char* file, int line);

#define CG_CUDA(call)                                                      \
  do {                                                                     \
    cudaError_t cg_e_ = (call);                                            \
    if (cg_e_ != cudaSuccess)                                              \
      return ::cg::cuda_fail(cg_e_, #call, __FILE__, __LINE__);            \
  } while (0)

#define CG_LAUNCH_CHECK()                                                  \
  do {                                                                     \
    cudaError_t cg_e_ = cudaGetLastError();                                \
    if (cg_e_ != cudaSuccess)                                              \
      return ::cg::cuda_fail(cg_e_, "kernel launch", __FILE__, __LINE__);  \
  } while (0)

#define CG_ARG(cond, ...)                                                  \
  do {                                                                     \
    if (!(cond)) {                                                         \
      ::cg::set_error(__VA_ARGS__);                                        \
      return CG_ERR_INVALID_ARG;                                           \
    }                                                                      \
  } while (0)

#define CG_TRY(expr)                                                       \
  do {                                                                     \
    int cg_s_ = (expr);                                                    \
    if (cg_s_ != CG_OK) return cg_s_;                                      \
  } while (0)

struct DeviceInfo {
  int device;
  int sm_count;
  size_t l2_bytes;
  size_t smem_optin;
};
// Properties of the current device (cached per device).
int device_info(DeviceInfo* out);

inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Grid size for grid-stride kernels: a multiple of the SM count.
int grid_for(int64_t n, int threads, int per_sm = 8);

// Stream-ordered scratch, given back when it goes out of scope.  Taken in
// slabs: an allocation from the stream-ordered pool costs 10-60 us of host
// time after every synchronisation (the pool gives its memory back then), and
// a build wants dozens of arrays.  `first` sizes the first slab.
struct Scratch {
  std::vector<void*> slabs;
  cudaStream_t s;
  size_t first;
  char* cur = nullptr;
  size_t left = 0;
  explicit Scratch(cudaStream_t st, size_t first_slab = 0) : s(st), first(first_slab) {}
  // over a buffer that a handle or a caller keeps, where it is not too small
  Scratch(cudaStream_t st, void* buffer, size_t bytes, size_t first_slab = 0)
      : s(st), first(first_slab) {
    if (bytes >= first_slab) {
      cur = static_cast<char*>(buffer);
      left = bytes;
    }
  }
  Scratch(const Scratch&) = delete;
  Scratch& operator=(const Scratch&) = delete;
  static size_t round(size_t b) { return (b + 255) & ~(size_t)255; }
  template <typename T>
  cudaError_t get(T** p, size_t n) {
    const size_t b = round(sizeof(T) * (n > 0 ? n : 1));
    if (b > left) {
      const size_t slab = b > first ? b : first;
      void* q = nullptr;
      cudaError_t e = cudaMallocAsync(&q, slab, s);
      if (e != cudaSuccess) return e;
      slabs.push_back(q);
      cur = static_cast<char*>(q);
      left = slab;
      first = (size_t)1 << 20;  // a slab that was sized too small goes on in small ones
    }
    *p = reinterpret_cast<T*>(cur);
    cur += b;
    left -= b;
    return cudaSuccess;
  }
  ~Scratch() {
    for (void* p : slabs) cudaFreeAsync(p, s);
  }
};

// ---------------------------------------------------------------------------
// Scans and sorts (scan.cu).  All stream-ordered; scratch from ws, or of their
// own.  scan_scratch / sort_scratch: the bytes they take for n items.
// ---------------------------------------------------------------------------
// out[i] = sum_{j<i} in[j] for i in [0, n]; out has n+1 entries.
int exclusive_scan_i64(const int64_t* in, int64_t* out, int64_t n, cudaStream_t s,
                       Scratch* ws = nullptr);
int exclusive_scan_i32_to_i64(const int32_t* in, int64_t* out, int64_t n, cudaStream_t s,
                              Scratch* ws = nullptr);
size_t scan_scratch(int64_t n);
size_t sort_scratch(int64_t n);
// Stable LSD radix sort of (key, value) pairs on the low `bits` bits of key.
int radix_sort_pairs(const uint32_t* keys_in, const int32_t* vals_in,
                     uint32_t* keys_out, int32_t* vals_out, int64_t n, int bits,
                     cudaStream_t s, Scratch* ws = nullptr);

// ---------------------------------------------------------------------------
// Chained launches (programmatic dependent launch): the blocks of a kernel
// launched with launch_chained are set up as soon as the blocks of the one
// before it in the stream have exited; chain_begin(), which every such kernel
// calls before it reads or writes memory, then waits until that one's writes
// are visible.  The order of execution is the stream's; what goes is the drain
// and the launch between two kernels, 2-3 us of each of an iteration's two to
// four (20 iterations at 20,011 vertices: 418 us without, 311 with; at 1 M 1393 and
// 1226, when this came; 1083 with what has changed since).  The next kernel is not let in earlier than that
// (griddepcontrol.launch_dependents): its waiting blocks then hold registers
// and shared memory, and with them L1, that the running kernel still wants
// (1835 us at 1 M vertices; 27.1 ms instead of 19.1 at 32 M).
// The blocks of such a kernel exist before the kernel in front of it has ended, so
// nothing that they read counts as read-only for as long as they run: they take no
// read-only-path load (__ldg, or what the compiler makes of a __restrict__
// pointer), but plain ones (__ldca, __ldcs, __ldcg).
// ---------------------------------------------------------------------------
template <typename... P, typename... A>
int launch_chained(void (*kernel)(P...), unsigned grid, unsigned threads, size_t smem,
                   cudaStream_t s, A... args) {
  cudaLaunchAttribute at{};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  CG_CUDA(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
  return CG_OK;
}

// Waits until a kernel on the stream has written the ticket to a pinned word:
// the host watches the word (a copy and a synchronisation take 17 us), asks the
// stream now and then whether it has failed, and sleeps in between when the wait
// gets long.
int wait_ticket(const unsigned long long* word, unsigned long long ticket, cudaStream_t s,
                const char* what);

// ---------------------------------------------------------------------------
// Device helpers
// ---------------------------------------------------------------------------
// Always true, which only the machine knows: what stands behind
// `if (!chain_begin()) return;` is not moved in front of it.
__device__ __forceinline__ bool chain_begin() {
  unsigned go;
  asm volatile("griddepcontrol.wait;\n\tmov.u32 %0, 1;" : "=r"(go)::"memory");
  return go != 0u;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  return v;
}

// Block-wide sum (result valid in thread 0).  `sh` holds >= 32 entries.
template <typename T, int THREADS>
__device__ __forceinline__ T block_sum(T v, T* sh) {
  v = warp_sum(v);
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  if (lane == 0) sh[w] = v;
  __syncthreads();
  T r = 0;
  if (w == 0) {
    r = lane < THREADS / 32 ? sh[lane] : T(0);
    r = warp_sum(r);
  }
  __syncthreads();
  return r;
}

// Streaming (evict-first) loads for data read once per pass.
template <typename T>
__device__ __forceinline__ T ld_stream(const T* p) { return __ldcs(p); }

}  // namespace cg
