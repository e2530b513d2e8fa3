// Shared by the fp32-FMA weight passes (zo_wpass_fma.cu, zo_wpass_gemm.cu): 16-byte vectors
// of W, its scalar access at ragged edges, asynchronous copies into shared memory, and the
// matrix of a tile.
#pragma once

#include "zo_kernels.h"

namespace zo {
namespace fma {

template <typename T> struct Vec;
template <> struct Vec<float> { static constexpr int N = 4; };
template <> struct Vec<__nv_bfloat16> { static constexpr int N = 8; };

template <typename T>
__device__ __forceinline__ float load_scalar(const T* p);
template <>
__device__ __forceinline__ float load_scalar<float>(const float* p) { return *p; }
template <>
__device__ __forceinline__ float load_scalar<__nv_bfloat16>(const __nv_bfloat16* p) {
  return __bfloat162float(*p);
}
template <typename T>
__device__ __forceinline__ void store_scalar(T* p, float x);
template <>
__device__ __forceinline__ void store_scalar<float>(float* p, float x) { *p = x; }
template <>
__device__ __forceinline__ void store_scalar<__nv_bfloat16>(__nv_bfloat16* p, float x) {
  *p = __float2bfloat16_rn(x);
}

__device__ __forceinline__ uint32_t pack2_bf16(float lo, float hi) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(lo, hi);   // RNE, lo in the low half
  return *reinterpret_cast<const uint32_t*>(&h);
}

// 16 bytes from global to shared memory without passing through registers; the bytes past
// src_bytes (0 .. 16) are zero-filled and not read.
__device__ __forceinline__ void cp_async_16(void* dst, const void* src, int src_bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_4(void* dst, const void* src, int src_bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src), "r"(src_bytes) : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;\n" ::: "memory");
}
template <int kPending>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(kPending) : "memory");
}

// The matrix whose tiles hold `tile`: the last i < n_mats with prefix[i] <= tile.  The 32
// lanes of each (full) warp probe 32 places at once, so a set of up to 1024 matrices takes
// two dependent loads; a binary search takes one per halving (eight for 224 matrices).
__device__ __forceinline__ int find_matrix(const int64_t* __restrict__ prefix, int n_mats,
                                           int64_t tile) {
  const int lane = threadIdx.x & 31;
  int lo = 0, n = n_mats;                        // candidates [lo, lo + n)
  while (n > 1) {
    const int step = (n + 31) / 32;
    const int i = lo + lane * step;
    const bool le = lane * step < n && __ldg(prefix + i) <= tile;
    const int k = 31 - __clz((int)__ballot_sync(0xffffffffu, le));   // lane 0 always holds
    lo += k * step;
    n = min(step, n - k * step);
  }
  return lo;
}

}  // namespace fma
}  // namespace zo
