// Host-side helpers: status strings, thread-local error text, device info.
#include <stdarg.h>

#include <chrono>
#include <mutex>
#include <thread>

#include "common.cuh"

namespace cg {

static thread_local char g_err[1024] = "";

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
}

const char* last_error() { return g_err; }

int cuda_fail(cudaError_t e, const char* what, const char* file, int line) {
  set_error("%s failed at %s:%d: %s (%s)", what, file, line, cudaGetErrorName(e),
            cudaGetErrorString(e));
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();  // clear the sticky-free allocation error
    return CG_ERR_OOM;
  }
  return CG_ERR_CUDA;
}

int device_info(DeviceInfo* out) {
  static std::mutex mu;
  static DeviceInfo cache[64];
  static bool have[64] = {false};
  int dev = 0;
  CG_CUDA(cudaGetDevice(&dev));
  if (dev < 0 || dev >= 64) {
    set_error("device ordinal %d out of range", dev);
    return CG_ERR_UNSUPPORTED;
  }
  std::lock_guard<std::mutex> lk(mu);
  if (!have[dev]) {
    DeviceInfo d{};
    d.device = dev;
    int v = 0;
    CG_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
    d.sm_count = v;
    CG_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrL2CacheSize, dev));
    d.l2_bytes = (size_t)v;
    CG_CUDA(cudaDeviceGetAttribute(&v, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
    d.smem_optin = (size_t)v;
    cache[dev] = d;
    have[dev] = true;
  }
  *out = cache[dev];
  return CG_OK;
}

int grid_for(int64_t n, int threads, int per_sm) {
  DeviceInfo di{};
  int sms = 148;
  if (device_info(&di) == CG_OK) sms = di.sm_count;
  int64_t want = ceil_div(n > 0 ? n : 1, threads);
  int64_t cap = (int64_t)sms * per_sm;
  return (int)(want < cap ? want : cap);
}

int wait_ticket(const unsigned long long* word, unsigned long long ticket, cudaStream_t s,
                const char* what) {
  using clock = std::chrono::steady_clock;
  const clock::time_point start = clock::now();
  for (unsigned spins = 1;; ++spins) {
    if (__atomic_load_n(word, __ATOMIC_ACQUIRE) == ticket) return CG_OK;
    if (spins % 4096) continue;
    const cudaError_t e = cudaStreamQuery(s);
    if (e == cudaSuccess) {  // all done: the word is there, or will never be
      if (__atomic_load_n(word, __ATOMIC_ACQUIRE) == ticket) return CG_OK;
      set_error("%s: a result did not reach the host", what);
      return CG_ERR_CUDA;
    }
    if (e != cudaErrorNotReady) return cuda_fail(e, what, __FILE__, __LINE__);
    // a long wait (other work in front of it on the stream) leaves the core to
    // others: from 5 ms on, sleeps of a 64th of the time waited so far
    const clock::duration waited = clock::now() - start;
    if (waited > std::chrono::milliseconds(5)) std::this_thread::sleep_for(waited / 64);
  }
}

}  // namespace cg

extern "C" {

const char* cg_status_string(int status) {
  switch (status) {
    case CG_OK: return "CG_OK";
    case CG_ERR_INVALID_ARG: return "CG_ERR_INVALID_ARG";
    case CG_ERR_OOM: return "CG_ERR_OOM";
    case CG_ERR_CUDA: return "CG_ERR_CUDA";
    case CG_ERR_TIMEOUT: return "CG_ERR_TIMEOUT";
    case CG_ERR_UNSUPPORTED: return "CG_ERR_UNSUPPORTED";
    default: return "CG_ERR_UNKNOWN";
  }
}

const char* cg_last_error_message(void) { return cg::last_error(); }

int cg_version(void) { return 100; }

}  // extern "C"
