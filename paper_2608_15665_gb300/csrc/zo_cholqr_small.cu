// Subspace refresh of fp32 weights at r = 4 and 8: Alg. 1's Haar factor of every panel in one
// launch, the panel held in registers.
//
// Tall panels (rows >= 4 r, at most 8 CTAs' worth) by CholeskyQR2 as in zo_cholqr.cu -- the
// unique Q with diag(R) > 0 of Eq. (11), twice Q <- X L^-T with L L^T = X^T X -- by one
// CTA or a cluster of up to eight: a thread draws its rows of Omega, both Gram matrices are
// sums over the CTA's threads (and, through distributed shared memory, the cluster's CTAs, in
// rank order), every thread factors the r x r matrix for itself and solves its rows in place.
// Panels shorter than 4 r (a LoRA factor's short side), whose condition number may be large,
// by one warp's Householder reflections, a row per lane, in the same launch.  The others
// (longer than the clusters hold) keep the TSQR of zo_qr.cu.
//
// Bound: latency.  The TSQR took three launches of dependent reflector steps for the LoRA set
// (160 panels of 5120 x 4 and 160 of 8 x 4: 46 + 29 + 24 us); here Omega's draws, two
// reductions and two r x r factorisations remain.
#include <algorithm>

#include "zo_cluster.cuh"
#include "zo_kernels.h"
#include "zo_launch.cuh"
#include "zo_reduce.cuh"

namespace zo {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// Rows per thread: about the most that 128 registers (two CTAs per SM) hold, because a panel that
// fits fewer CTAs needs fewer exchanges, and one that fits no cluster falls back to the TSQR.  At
// r = 4 20 rows spill 32 bytes, 22 564; at r = 8 8 rows spill none, 10 96 and 12 232.  A refresh of
// 160 fp32 matrices 8 x L in us (one 8 x 8192 matrix alone 16.6 with 20 rows, 14.4 with 10):
//   r = 4, L =   1024   4096   5120   8192  11008  16384  20480  32768  40960
//     10 rows     8.3   22.6   22.6   30.8   45.1   51.2   55.4    163    201
//     16 rows    10.3   16.5   24.7   29.0   37.5   43.1   60.5     75    201
//     20 rows    10.3   16.5   18.5   30.8   39.9   45.8   51.4     84     95
//     22 rows    10.3   18.5   20.6   32.8   36.9   47.9   53.9     88     98
//   r = 8
//      4 rows    12.4   41.2   59.7   66.8    164    195    236    356    433
//      8 rows    14.9   39.0   47.9   55.8     85     97    238    356    433
//     10 rows    16.7   41.0   43.1   58.8     92    103    113    356    433
template <int R>
struct SmallShape {
  static constexpr int kRPT = R == 4 ? 20 : 8;             // rows per thread
  static constexpr int kRows = kThreads * kRPT;            // rows per CTA
  static constexpr int kSums = R * (R + 1) / 2;            // the lower triangle, packed by rows
  static constexpr int kPad = R == 4 ? 16 : 64;
};
__host__ __device__ constexpr int tri(int i, int j) { return i * (i + 1) / 2 + j; }

__device__ __forceinline__ float ld_cluster(const float* p, uint32_t rank) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cta2::map_to(p, rank)) : "memory");
  return v;
}

// A row of Omega: the packed transform for tall panels; CUDA's functions for short ones, whose
// condition number can turn a last place into 1e-5 of Q.
template <int R, bool kTall>
__device__ __forceinline__ void draw_row(const CqPanel& pn, int64_t row, uint64_t seed,
                                         uint32_t refresh_idx, float (&x)[R]) {
#pragma unroll
  for (int c4 = 0; c4 < R / 4; ++c4) {
    const uint32_t c = (uint32_t)(row * (R / 4) + c4);
    const float4 z = kTall ? normal4_packed(seed, c, pn.gidx, refresh_idx, query_word(pn.tag, 0))
                           : normal4(seed, c, pn.gidx, refresh_idx, query_word(pn.tag, 0));
    x[4 * c4] = z.x; x[4 * c4 + 1] = z.y; x[4 * c4 + 2] = z.z; x[4 * c4 + 3] = z.w;
  }
}
template <int R>
__device__ __forceinline__ void store_row(const CqPanel& pn, int64_t row, const float (&x)[R]) {
  float4* out = reinterpret_cast<float4*>(pn.out + row * R);
#pragma unroll
  for (int c4 = 0; c4 < R / 4; ++c4)
    out[c4] = make_float4(x[4 * c4], x[4 * c4 + 1], x[4 * c4 + 2], x[4 * c4 + 3]);
}

// One panel of at most 32 rows by one warp: Householder with row i in lane i (the convention,
// sums and bits of zo_qr.cu), then Q = H_0 ... H_(R-1) [diag(sgn R_cc); 0], sgn(0) = +1.
template <int R>
__device__ __forceinline__ void short_panel(const CqPanel& pn, uint64_t seed, uint32_t refresh_idx) {
  const int lane = threadIdx.x & 31;
  const bool live = lane < (int)pn.rows;
  float a[R];
#pragma unroll
  for (int c = 0; c < R; ++c) a[c] = 0.f;
  if (live) draw_row<R, false>(pn, lane, seed, refresh_idx, a);
  float tau[R], diag[R];
#pragma unroll
  for (int j = 0; j < R; ++j) {
    // sums over the rows below j of a_ij a_ic, c >= j
    float p[R], rowj[R];
#pragma unroll
    for (int c = j; c < R; ++c) {
      p[c] = lane > j ? a[j] * a[c] : 0.f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) p[c] += __shfl_xor_sync(0xffffffffu, p[c], o);
      rowj[c] = __shfl_sync(0xffffffffu, a[c], j);
    }
    const float alpha = rowj[j];
    float t = 0.f, beta = alpha, scale = 0.f;
    if (p[j] != 0.f) {
      beta = -copysignf(sqrtf(fmaf(alpha, alpha, p[j])), alpha);
      t = (beta - alpha) / beta;
      scale = 1.0f / (alpha - beta);
    }
    tau[j] = t;
    diag[j] = beta;
    const float v = lane == j ? 1.f : a[j] * scale;
#pragma unroll
    for (int c = j + 1; c < R; ++c)
      if (lane >= j) a[c] = fmaf(-t * v, fmaf(scale, p[c], rowj[c]), a[c]);
    a[j] = lane > j ? v : a[j];              // the reflector over the eliminated column
  }
  float q[R];
#pragma unroll
  for (int c = 0; c < R; ++c) q[c] = lane == c ? (diag[c] < 0.f ? -1.f : 1.f) : 0.f;
#pragma unroll
  for (int j = R - 1; j >= 0; --j) {
    const float v = lane < j ? 0.f : lane == j ? 1.f : a[j];
#pragma unroll
    for (int c = 0; c < R; ++c) {
      float p = v * q[c];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) p += __shfl_xor_sync(0xffffffffu, p, o);
      q[c] = fmaf(-tau[j] * v, p, q[c]);
    }
  }
  if (live) store_row<R>(pn, lane, q);
}

// Grid: `ctas` CTAs for each of the n_tall panels (clusters of that size), then, with ctas = 1,
// a CTA for every eight of the n_short short ones.
template <int R>
__global__ void __launch_bounds__(kThreads, 2)
cq_small_kernel(const CqPanel* __restrict__ tall, int n_tall, const CqPanel* __restrict__ shorts,
                int n_short, int ctas, uint64_t seed, uint32_t refresh_idx,
                uint32_t* __restrict__ status) {
  using S = SmallShape<R>;
  __shared__ float red[kWarps][S::kPad];
  __shared__ float part[2][S::kSums];        // this CTA's sums of either round
  __shared__ float G[S::kSums];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int which = (int)(blockIdx.x / ctas), rank = (int)(blockIdx.x % ctas);
  if (which >= n_tall) {
    const int k = (which - n_tall) * kWarps + warp;
    if (k < n_short) short_panel<R>(shorts[k], seed, refresh_idx);
    return;
  }
  const CqPanel pn = tall[which];
  float x[S::kRPT][R];
#pragma unroll
  for (int k = 0; k < S::kRPT; ++k) {
    const int64_t row = (int64_t)(k * ctas + rank) * kThreads + tid;
#pragma unroll
    for (int c = 0; c < R; ++c) x[k][c] = 0.f;
    if (row < pn.rows) draw_row<R, true>(pn, row, seed, refresh_idx, x[k]);
  }
  bool bad = false;
#pragma unroll 1
  for (int round = 0; round < 2; ++round) {
    float p[S::kPad];
#pragma unroll
    for (int e = 0; e < S::kPad; ++e) p[e] = 0.f;
#pragma unroll
    for (int k = 0; k < S::kRPT; ++k)
#pragma unroll
      for (int i = 0; i < R; ++i)
#pragma unroll
        for (int j = 0; j <= i; ++j) p[tri(i, j)] = fmaf(x[k][i], x[k][j], p[tri(i, j)]);
    warp_reduce_scatter<S::kPad>(p, lane);
    if constexpr (S::kPad >= 32) {
#pragma unroll
      for (int k = 0; k < S::kPad / 32; ++k) red[warp][lane * (S::kPad / 32) + k] = p[k];
    } else {
      if (lane % (32 / S::kPad) == 0) red[warp][lane / (32 / S::kPad)] = p[0];
    }
    __syncthreads();
    if (tid < S::kSums) {
      float s = 0.f;
#pragma unroll
      for (int w = 0; w < kWarps; ++w) s += red[w][tid];
      if (ctas == 1) G[tid] = s;
      else part[round][tid] = s;
    }
    if (ctas > 1) {
      cta2::cluster_sync_all();
      if (tid < S::kSums) {
        float s = 0.f;
        for (int c = 0; c < ctas; ++c) s += ld_cluster(&part[round][tid], (uint32_t)c);
        G[tid] = s;
      }
    }
    __syncthreads();
    // G = L L^T, for every thread alike; then each row x <- x L^-T by forward substitution
    float g[S::kSums], inv[R];
#pragma unroll
    for (int e = 0; e < S::kSums; ++e) g[e] = G[e];
#pragma unroll
    for (int j = 0; j < R; ++j) {
      const float d = g[tri(j, j)];
      bad = bad || !(d > 0.f);
      inv[j] = 1.0f / sqrtf(d > 0.f ? d : 1.f);
#pragma unroll
      for (int i = j + 1; i < R; ++i) g[tri(i, j)] *= inv[j];
#pragma unroll
      for (int i = j + 1; i < R; ++i)
#pragma unroll
        for (int k = j + 1; k <= i; ++k)
          g[tri(i, k)] = fmaf(-g[tri(i, j)], g[tri(k, j)], g[tri(i, k)]);
    }
#pragma unroll
    for (int k = 0; k < S::kRPT; ++k)
#pragma unroll
      for (int c = 0; c < R; ++c) {
        float q = x[k][c];
#pragma unroll
        for (int b = 0; b < c; ++b) q = fmaf(-g[tri(c, b)], x[k][b], q);
        x[k][c] = q * inv[c];
      }
  }
#pragma unroll
  for (int k = 0; k < S::kRPT; ++k) {
    const int64_t row = (int64_t)(k * ctas + rank) * kThreads + tid;
    if (row < pn.rows) {
      if (bad) {
#pragma unroll
        for (int c = 0; c < R; ++c) x[k][c] = 0.f;
      }
      store_row<R>(pn, row, x[k]);
    }
  }
  if (bad && rank == 0 && tid == 0) atomicOr(status, (uint32_t)kDevNotPosDef);
  if (ctas > 1) cta2::cluster_sync_all();    // the peers have read this CTA's sums
}

template <int R>
cudaError_t launch_small_r(const CqPanel* tall, int n_tall, const CqPanel* shorts, int n_short,
                           int ctas, uint64_t seed, uint32_t refresh_idx, uint32_t* d_status,
                           cudaStream_t s) {
  const unsigned grid = (unsigned)(n_tall * ctas + (n_short + kWarps - 1) / kWarps);
  return launch_dependent(cq_small_kernel<R>, grid, kThreads, 0, s, (unsigned)ctas,
                          /*dependent=*/false, tall, n_tall, shorts, n_short, ctas, seed, refresh_idx,
                          d_status);
}

}  // namespace

int32_t cholqr_small_ctas(int32_t r, int64_t rows) {
  const int64_t per = r == 4 ? SmallShape<4>::kRows : r == 8 ? SmallShape<8>::kRows : 0;
  if (per == 0 || rows < 4 * (int64_t)r) return 0;
  for (int32_t c = 1; c <= 8; c *= 2)
    if (rows <= per * c) return c;
  return 0;
}

bool cholqr_small_short(int32_t r, int64_t rows) { return (r == 4 || r == 8) && rows < 4 * (int64_t)r; }

cudaError_t launch_cholqr_small(const CqPanel* d_tall, int32_t n_tall, const CqPanel* d_short,
                                int32_t n_short, int32_t ctas, int32_t r, uint64_t seed,
                                uint32_t refresh_idx, uint32_t* d_status, cudaStream_t s) {
  if (n_tall <= 0 && n_short <= 0) return cudaSuccess;
  if (n_short > 0 && ctas != 1) return cudaErrorInvalidValue;
  if (r == 4)
    return launch_small_r<4>(d_tall, n_tall, d_short, n_short, ctas, seed, refresh_idx, d_status, s);
  if (r == 8)
    return launch_small_r<8>(d_tall, n_tall, d_short, n_short, ctas, seed, refresh_idx, d_status, s);
  return cudaErrorInvalidValue;
}

}  // namespace zo
