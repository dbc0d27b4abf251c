// Factor storage of collaborative filtering: FP32, BF16, or BF16 hi + lo.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace cg {
namespace {

__device__ __forceinline__ float b_lo(uint32_t w) { return __uint_as_float(w << 16); }
__device__ __forceinline__ float b_hi(uint32_t w) { return __uint_as_float(w & 0xffff0000u); }

// BF16 hi + lo is stored as one 32-bit word per dimension (hi in the low
// half, lo in the high half), so a row has the size of an FP32 row.
__device__ __forceinline__ float hilo(uint32_t w) { return b_lo(w) + b_hi(w); }

// Entries [at, at + 4) (at a multiple of 4) as stored, and as FP32.
template <int PREC>
__device__ __forceinline__ uint4 raw4(const void* p0, int64_t at) {
  if (PREC == 1) {
    const uint2 h = __ldg(reinterpret_cast<const uint2*>(static_cast<const uint16_t*>(p0) + at));
    return make_uint4(h.x, h.y, 0u, 0u);
  }
  return __ldg(reinterpret_cast<const uint4*>(static_cast<const uint32_t*>(p0) + at));
}
template <int PREC>
__device__ __forceinline__ float4 decode4(const uint4& h) {
  if (PREC == 0)
    return make_float4(__uint_as_float(h.x), __uint_as_float(h.y), __uint_as_float(h.z),
                       __uint_as_float(h.w));
  if (PREC == 1) return make_float4(b_lo(h.x), b_hi(h.x), b_lo(h.y), b_hi(h.y));
  return make_float4(hilo(h.x), hilo(h.y), hilo(h.z), hilo(h.w));
}
template <int PREC>
__device__ __forceinline__ float4 load4(const void* p0, int64_t at) {
  return decode4<PREC>(raw4<PREC>(p0, at));
}

}  // namespace
}  // namespace cg
