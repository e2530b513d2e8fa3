// Pieces shared by the perturbed-linear GEMM files (zo_linear.cu: single-CTA tiles and the
// S = X P^T kernel; zo_linear_pair.cu: SM-pair tiles, zo_linear_few.cu: tiles of few tokens,
// both with S computed in-kernel).
#pragma once

#include <cuda_bf16.h>
#include <cstdint>

#include "zo_tc_common.cuh"

namespace zo {
namespace lin {

// Ready flags of S_HL rows: each writer sets its own to the call's epoch.
__device__ __forceinline__ void set_ready(uint32_t* f, uint32_t epoch) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(f), "r"(epoch) : "memory");
}
// every one of the n (<= 32) flags at f holds epoch (bounded; false on abort or timeout).
// Each poll issues the n loads together (relaxed, independent, so they overlap in one L2
// round trip -- acquire loads would complete one after another); once all match, one
// acquire-release fence gives the acquire.
__device__ __forceinline__ bool wait_s_rows(const uint32_t* f, int n, uint32_t epoch,
                                            const volatile int* abort, long long limit_cycles) {
  const long long t0 = clock64();
  for (;;) {
    uint32_t v[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      v[j] = epoch;
      if (j < n)
        asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v[j]) : "l"(f + j) : "memory");
    }
    bool all = true;
#pragma unroll
    for (int j = 0; j < 32; ++j) all = all && v[j] == epoch;
    if (all) {
      asm volatile("fence.acq_rel.gpu;" ::: "memory");
      return true;
    }
    if (*abort) return false;
    if (clock64() - t0 > limit_cycles) return false;
    __nanosleep(64);
  }
}
// generic-proxy global writes <-> later async-proxy (TMA) reads
__device__ __forceinline__ void fence_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}

// An S_HL row holds hl_width(R) bf16: [hi | lo] of the R sums in groups of 8, then zeros
// (R = 16).  write_s_chunk: the hi and lo groups of sums kC j .. kC j + kC - 1, kC =
// min(R, 32).
template <int R>
__device__ __forceinline__ void write_s_chunk(__nv_bfloat16* s_hl, int row, int j,
                                              const float (&x)[R < 32 ? R : 32]) {
  constexpr int kC = R < 32 ? R : 32;
  uint4* out = reinterpret_cast<uint4*>(s_hl + (int64_t)row * tc::hl_width(R));
#pragma unroll
  for (int g = 0; g < kC / 8; ++g) {
    float c[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) c[e] = x[8 * g + e];
    uint4 hi, lo;
    tc::split8(c, hi, lo);
    out[kC / 8 * j + g] = hi;
    out[R / 8 + kC / 8 * j + g] = lo;
  }
}

// the zero groups of an S_HL row past 2R
template <int R>
__device__ __forceinline__ void zero_s_pad(__nv_bfloat16* s_hl, int row) {
  uint4* out = reinterpret_cast<uint4*>(s_hl + (int64_t)row * tc::hl_width(R));
#pragma unroll
  for (int z = R / 4; z < tc::hl_width(R) / 8; ++z) out[z] = make_uint4(0u, 0u, 0u, 0u);
}

// a whole S_HL row, R <= 32
template <int R>
__device__ __forceinline__ void write_s_row(__nv_bfloat16* s_hl, int row, const float (&x)[R]) {
  static_assert(R <= 32, "one chunk per row");
  write_s_chunk<R>(s_hl, row, 0, x);
  zero_s_pad<R>(s_hl, row);
}

}  // namespace lin
}  // namespace zo
