// Subspace refresh: Alg. 1 (the Haar-distributed bases U, V) for every matrix in a few launches.
//
// For each panel (Omega_U, m x r and Omega_V, n x r) we need the thin QR factor
// with a positive diagonal of R (Eq. (11)).  Panels are tall and skinny (m up to
// 25600, r <= 128) and there are up to ~900 of them, so the factorisation is a
// batched TSQR (communication-avoiding QR, Demmel et al. 2012):
//
//   up pass, level 0:  each block of B rows draws its Omega rows from the
//                      counter contract, factors them by Householder reflections
//                      held in registers (one or more rows per thread), stores
//                      the reflectors over its rows and its r x r R factor into
//                      the next level's stack.
//   up pass, level l:  the stacked R factors are factored the same way.
//   top block:         once a panel's stack fits in one block, that block forms
//                      Q_top = H_0 ... H_(r-1) [diag(sgn R_cc); 0] directly -- the sign
//                      correction of Eq. (11) folded into the start of Q -- and
//                      writes it over its stack.
//   down pass:         every other block applies its reflectors to [S; 0], S the
//                      r x r block of its parent's Q that multiplies its R, giving
//                      its rows of Q; at level 0 those are the rows of U (or V).
//
// Householder convention (Golub & Van Loan, Sec. 5.1): for x = A[j:, j],
// beta = -sign(x_0) ||x||, v = x / (x_0 - beta) with v_0 = 1, tau = (beta - x_0)/beta.
// Blocks with fewer real rows than B are padded with zero rows, which leaves the
// factorisation of the real rows unchanged and produces zero rows of Q there.
#include "zo_kernels.h"
#include "zo_reduce.cuh"

namespace zo {
namespace {

constexpr int kQrThreads = 256;
constexpr int kQrWarps = kQrThreads / 32;

template <int R>
struct QrShape {
  static constexpr int kRPT = R >= 64 ? 1 : 64 / R;   // rows per thread
  static constexpr int kB = kQrThreads * kRPT;        // rows per block
  static constexpr int kLd = R + 1;                   // padded row stride of the reflector copy
};

// Shared scratch of one QR block.
template <int R>
struct QrSmem {
  float red[2][kQrWarps][R];   // per-warp partial sums, double-buffered by step parity
  float wbuf[2][R];            // reduced vector of the current step
  float rowj[2][R];            // row j of the panel (owner's copy)
  float scal[2][2];            // tau, 1/(alpha - beta) of the current step
  float diag[R];               // beta_j = R_jj
  float tau[R];
};

// A step's columns in groups: a group left of the step's column is passed over by all threads
// alike, and the 32 (or R) columns of a set are reduced together.
template <int R>
struct QrCols {
  static constexpr int kG = R < 16 ? R : 16;
  static constexpr int kH = R < 32 ? R : 32;
  static constexpr int kC32 = (R + 31) / 32;       // 32-column groups handled by warp 0
};

// Block-wide sums of a set's per-thread values: one partial per warp to red[0 .. H - 1].
template <int H>
__device__ __forceinline__ void warp_partials(float (&p)[H], float* red) {
  const int lane = threadIdx.x & 31;
  warp_reduce_scatter<H>(p, lane);
  if (lane % (32 / H) == 0) red[lane / (32 / H)] = p[0];
}

// Householder factorisation of the block held in registers (row i = rho*256 + tid); rows from
// n_real on are zero.
//
// Bound: instruction issue and two barriers per column.  The column's own entry comes from its
// group (or, at r <= 16, where the columns are unrolled, from a fixed register), groups left of
// the column and warps without rows below it take no part: a shorter panel or a later column
// costs less, and every remaining sum is the same.  8 pairs of panels of 200 x 64: 283 -> 158 us a
// refresh, of 400 and 504 x 128: 2497 -> 1142; 24 layers of the 1.3B set at r = 4: 78 -> 60, at
// r = 8: 147 -> 86.
template <int R>
__device__ void factor_block(float (&a)[QrShape<R>::kRPT][R], int n_real, QrSmem<R>& sm) {
  constexpr int RPT = QrShape<R>::kRPT;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  using Qc = QrCols<R>;
  constexpr int kG = Qc::kG, kH = Qc::kH;
  const int last = (RPT - 1) * kQrThreads + 32 * warp + 31;     // the warp's last row
  const bool real = 32 * warp < n_real;
#pragma unroll (R <= 16 ? R : 1)
  for (int j = 0; j < R; ++j) {
    const int buf = j & 1;
    float xj[RPT];
#pragma unroll
    for (int rho = 0; rho < RPT; ++rho) xj[rho] = 0.f;
    if (real && last >= j) {
#pragma unroll
      for (int g = 0; g < R / kG; ++g)
        if (g * kG + kG > j)
#pragma unroll
          for (int c = 0; c < kG; ++c)
#pragma unroll
            for (int rho = 0; rho < RPT; ++rho)
              xj[rho] = g * kG + c == j ? a[rho][g * kG + c] : xj[rho];
    }
#pragma unroll
    for (int hh = 0; hh < R / kH; ++hh) {
      if (hh * kH + kH <= j) continue;
      float* red = &sm.red[buf][warp][hh * kH];
      if (!real || last <= j) {
        if (lane < kH) red[lane] = 0.f;
        continue;
      }
      float p[kH];
#pragma unroll
      for (int c = 0; c < kH; ++c) p[c] = 0.f;
#pragma unroll
      for (int rho = 0; rho < RPT; ++rho) {
        if (rho * kQrThreads + tid <= j) continue;
#pragma unroll
        for (int g = 0; g < kH / kG; ++g) {
          if (hh * kH + g * kG + kG <= j) continue;
#pragma unroll
          for (int c = g * kG; c < g * kG + kG; ++c) p[c] = fmaf(xj[rho], a[rho][hh * kH + c], p[c]);
        }
      }
      warp_partials<kH>(p, red);
    }
    if (tid == j) {
#pragma unroll
      for (int c = 0; c < R; ++c) sm.rowj[buf][c] = a[0][c];
    }
    __syncthreads();
    if (warp == 0) {
      float sk[Qc::kC32];
#pragma unroll
      for (int k = 0; k < Qc::kC32; ++k) {
        const int c = lane + 32 * k;
        sk[k] = 0.f;
        if (c < R) {
#pragma unroll
          for (int w = 0; w < kQrWarps; ++w) sk[k] += sm.red[buf][w][c];
        }
      }
      float sel = 0.f;
#pragma unroll
      for (int k = 0; k < Qc::kC32; ++k)
        if (k == (j >> 5)) sel = sk[k];
      const float s_j = __shfl_sync(0xffffffffu, sel, j & 31);
      const float alpha = sm.rowj[buf][j];
      float tau = 0.f, beta = alpha, scale = 0.f;
      if (s_j != 0.f) {
        beta = -copysignf(sqrtf(fmaf(alpha, alpha, s_j)), alpha);
        tau = (beta - alpha) / beta;
        scale = 1.0f / (alpha - beta);
      }
#pragma unroll
      for (int k = 0; k < Qc::kC32; ++k) {
        const int c = lane + 32 * k;
        if (c < R && c > j) sm.wbuf[buf][c] = fmaf(scale, sk[k], sm.rowj[buf][c]);
      }
      if (lane == 0) {
        sm.scal[buf][0] = tau;
        sm.scal[buf][1] = scale;
        sm.diag[j] = beta;
        sm.tau[j] = tau;
      }
    }
    __syncthreads();
    if (!real || last < j) continue;
    const float tau = sm.scal[buf][0], scale = sm.scal[buf][1], beta = sm.diag[j];
#pragma unroll
    for (int rho = 0; rho < RPT; ++rho) {
      const int i = rho * kQrThreads + tid;
      if (i < j) continue;
      const float v = xj[rho] * scale;
      const float tv = i > j ? -tau * v : -tau;
#pragma unroll
      for (int g = 0; g < R / kG; ++g) {
        if (g * kG > j) {
#pragma unroll
          for (int c = g * kG; c < g * kG + kG; ++c)
            a[rho][c] = fmaf(tv, sm.wbuf[buf][c], a[rho][c]);
        } else if (g * kG + kG > j) {
#pragma unroll
          for (int c = g * kG; c < g * kG + kG; ++c) {
            if (c > j) a[rho][c] = fmaf(tv, sm.wbuf[buf][c], a[rho][c]);
            if (c == j) a[rho][c] = i > j ? v : beta;
          }
        }
      }
    }
  }
}

// Y <- H_0 H_1 ... H_(R-1) Y with the reflectors in refl (padded stride kLd).  upper: Y starts
// as a diagonal, so that the columns left of j are still zero from row j on.
template <int R>
__device__ void apply_reflectors_backward(float (&a)[QrShape<R>::kRPT][R], const float* refl,
                                          int n_real, bool upper, QrSmem<R>& sm) {
  constexpr int RPT = QrShape<R>::kRPT;
  constexpr int LD = QrShape<R>::kLd;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  using Qc = QrCols<R>;
  constexpr int kG = Qc::kG, kH = Qc::kH;
  const int last = (RPT - 1) * kQrThreads + 32 * warp + 31;
  const bool real = 32 * warp < n_real;
  for (int j = R - 1; j >= 0; --j) {
    const int buf = j & 1;
    const int c_min = upper ? j : 0;               // first column that changes
    float v[RPT];
#pragma unroll
    for (int rho = 0; rho < RPT; ++rho) {
      const int i = rho * kQrThreads + tid;
      v[rho] = i == j ? 1.0f : i > j ? refl[i * LD + j] : 0.f;
    }
#pragma unroll
    for (int hh = 0; hh < R / kH; ++hh) {
      if (hh * kH + kH <= c_min) continue;
      float* red = &sm.red[buf][warp][hh * kH];
      if (!real || last < j) {
        if (lane < kH) red[lane] = 0.f;
        continue;
      }
      float p[kH];
#pragma unroll
      for (int c = 0; c < kH; ++c) p[c] = 0.f;
#pragma unroll
      for (int rho = 0; rho < RPT; ++rho) {
        if (rho * kQrThreads + tid < j) continue;
#pragma unroll
        for (int g = 0; g < kH / kG; ++g) {
          if (hh * kH + g * kG + kG <= c_min) continue;
#pragma unroll
          for (int c = g * kG; c < g * kG + kG; ++c) p[c] = fmaf(v[rho], a[rho][hh * kH + c], p[c]);
        }
      }
      warp_partials<kH>(p, red);
    }
    __syncthreads();
    if (warp == 0) {
#pragma unroll
      for (int h = 0; h < Qc::kC32; ++h) {
        const int c = lane + 32 * h;
        if (c < R) {
          float s = 0.f;
#pragma unroll
          for (int w = 0; w < kQrWarps; ++w) s += sm.red[buf][w][c];
          sm.wbuf[buf][c] = s;
        }
      }
    }
    __syncthreads();
    if (!real || last < j) continue;
    const float tau = sm.tau[j];
#pragma unroll
    for (int rho = 0; rho < RPT; ++rho) {
      if (rho * kQrThreads + tid < j) continue;
      const float tv = -tau * v[rho];
#pragma unroll
      for (int g = 0; g < R / kG; ++g) {
        if (g * kG + kG <= c_min) continue;
#pragma unroll
        for (int c = g * kG; c < g * kG + kG; ++c)
          a[rho][c] = fmaf(tv, sm.wbuf[buf][c], a[rho][c]);
      }
    }
  }
}

template <int R>
__device__ __forceinline__ void store_rows(const float (&a)[QrShape<R>::kRPT][R], float* dst,
                                           int n_real) {
  constexpr int RPT = QrShape<R>::kRPT;
#pragma unroll
  for (int rho = 0; rho < RPT; ++rho) {
    const int i = rho * kQrThreads + threadIdx.x;
    if (i < n_real) {
      float4* d4 = reinterpret_cast<float4*>(dst + (int64_t)i * R);
#pragma unroll
      for (int c4 = 0; c4 < R / 4; ++c4)
        d4[c4] = make_float4(a[rho][4 * c4], a[rho][4 * c4 + 1], a[rho][4 * c4 + 2],
                             a[rho][4 * c4 + 3]);
    }
  }
}

template <int R>
__device__ __forceinline__ void regs_to_refl(const float (&a)[QrShape<R>::kRPT][R], float* refl) {
  constexpr int RPT = QrShape<R>::kRPT;
  constexpr int LD = QrShape<R>::kLd;
#pragma unroll
  for (int rho = 0; rho < RPT; ++rho) {
    const int i = rho * kQrThreads + threadIdx.x;
#pragma unroll
    for (int c = 0; c < R; ++c) refl[i * LD + c] = a[rho][c];
  }
}

template <int R>
__global__ void __launch_bounds__(kQrThreads)
qr_up_kernel(const QrBlock* __restrict__ blocks, uint64_t seed, uint32_t refresh_idx) {
  constexpr int RPT = QrShape<R>::kRPT;
  extern __shared__ float4 qr_smem4[];
  QrSmem<R>& sm = *reinterpret_cast<QrSmem<R>*>(qr_smem4);
  float* refl = reinterpret_cast<float*>(qr_smem4) + (sizeof(QrSmem<R>) + 15) / 16 * 4;
  const QrBlock blk = blocks[blockIdx.x];
  const int tid = threadIdx.x;

  float a[RPT][R];
#pragma unroll
  for (int rho = 0; rho < RPT; ++rho) {
    const int i = rho * kQrThreads + tid;
    if (i < blk.n_real) {
      if (blk.flags & kQrLevel0) {
        // element e = (row0 + i) * R + c of the panel uses counter e / 4, lane e % 4
        const uint32_t c0 = (uint32_t)(((blk.row0 + i) * R) >> 2);
#pragma unroll
        for (int c4 = 0; c4 < R / 4; ++c4) {
          const float4 z = normal4(seed, c0 + c4, blk.gidx, refresh_idx, query_word(blk.tag, 0));
          a[rho][4 * c4] = z.x; a[rho][4 * c4 + 1] = z.y;
          a[rho][4 * c4 + 2] = z.z; a[rho][4 * c4 + 3] = z.w;
        }
      } else {
        const float4* s4 = reinterpret_cast<const float4*>(blk.rows + (int64_t)i * R);
#pragma unroll
        for (int c4 = 0; c4 < R / 4; ++c4) {
          const float4 z = s4[c4];
          a[rho][4 * c4] = z.x; a[rho][4 * c4 + 1] = z.y;
          a[rho][4 * c4 + 2] = z.z; a[rho][4 * c4 + 3] = z.w;
        }
      }
    } else {
#pragma unroll
      for (int c = 0; c < R; ++c) a[rho][c] = 0.f;
    }
  }

  factor_block<R>(a, blk.n_real, sm);

  if (blk.flags & kQrTop) {
    regs_to_refl<R>(a, refl);
    __syncthreads();
    // Q = H_0 ... H_(R-1) [diag(sgn R_cc); 0]  (Eq. (11), sgn(0) = +1)
#pragma unroll
    for (int rho = 0; rho < RPT; ++rho) {
      const int i = rho * kQrThreads + tid;
#pragma unroll
      for (int c = 0; c < R; ++c) a[rho][c] = (i == c) ? (sm.diag[c] < 0.f ? -1.f : 1.f) : 0.f;
    }
    apply_reflectors_backward<R>(a, refl, blk.n_real, true, sm);
    store_rows<R>(a, blk.rows, blk.n_real);
  } else {
    store_rows<R>(a, blk.rows, blk.n_real);
    if (tid < R) {
      // R factor row `tid` (upper triangle of the block's first R rows)
      float4* d4 = reinterpret_cast<float4*>(blk.r_out + tid * R);
#pragma unroll
      for (int c4 = 0; c4 < R / 4; ++c4) {
        float v[4];
#pragma unroll
        for (int l = 0; l < 4; ++l) v[l] = (4 * c4 + l >= tid) ? a[0][4 * c4 + l] : 0.f;
        d4[c4] = make_float4(v[0], v[1], v[2], v[3]);
      }
      blk.tau[tid] = sm.tau[tid];
    }
  }
}

template <int R>
__global__ void __launch_bounds__(kQrThreads) qr_down_kernel(const QrBlock* __restrict__ blocks) {
  constexpr int RPT = QrShape<R>::kRPT;
  constexpr int LD = QrShape<R>::kLd;
  extern __shared__ float4 qr_smem4[];
  QrSmem<R>& sm = *reinterpret_cast<QrSmem<R>*>(qr_smem4);
  float* refl = reinterpret_cast<float*>(qr_smem4) + (sizeof(QrSmem<R>) + 15) / 16 * 4;
  const QrBlock blk = blocks[blockIdx.x];
  const int tid = threadIdx.x;

  float a[RPT][R];
#pragma unroll
  for (int rho = 0; rho < RPT; ++rho) {
    const int i = rho * kQrThreads + tid;
    if (i < blk.n_real) {
      const float4* s4 = reinterpret_cast<const float4*>(blk.rows + (int64_t)i * R);
#pragma unroll
      for (int c4 = 0; c4 < R / 4; ++c4) {
        const float4 z = s4[c4];
        refl[i * LD + 4 * c4] = z.x; refl[i * LD + 4 * c4 + 1] = z.y;
        refl[i * LD + 4 * c4 + 2] = z.z; refl[i * LD + 4 * c4 + 3] = z.w;
      }
    } else {
#pragma unroll
      for (int c = 0; c < R; ++c) refl[i * LD + c] = 0.f;
    }
    // Y = [S; 0]
#pragma unroll
    for (int c = 0; c < R; ++c) a[rho][c] = (i < R) ? blk.s_in[i * R + c] : 0.f;
  }
  if (tid < R) sm.tau[tid] = blk.tau[tid];
  __syncthreads();
  apply_reflectors_backward<R>(a, refl, blk.n_real, false, sm);
  store_rows<R>(a, blk.rows, blk.n_real);
}

template <int R>
size_t qr_smem_bytes() {
  return (sizeof(QrSmem<R>) + 15) / 16 * 16 +
         sizeof(float) * (size_t)QrShape<R>::kB * QrShape<R>::kLd;
}

template <int R>
cudaError_t launch_up_r(const QrBlock* d_blocks, int32_t n_blocks, uint64_t seed, uint32_t j,
                        cudaStream_t s) {
  const size_t smem = qr_smem_bytes<R>();
  cudaError_t e = cudaFuncSetAttribute(qr_up_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem);
  if (e != cudaSuccess) return e;
  qr_up_kernel<R><<<n_blocks, kQrThreads, smem, s>>>(d_blocks, seed, j);
  return cudaGetLastError();
}

template <int R>
cudaError_t launch_down_r(const QrBlock* d_blocks, int32_t n_blocks, cudaStream_t s) {
  const size_t smem = qr_smem_bytes<R>();
  cudaError_t e = cudaFuncSetAttribute(qr_down_kernel<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  qr_down_kernel<R><<<n_blocks, kQrThreads, smem, s>>>(d_blocks);
  return cudaGetLastError();
}

__global__ void zero_moments_kernel(const MatDesc* __restrict__ mats, int r) {
  const MatDesc md = mats[blockIdx.x];
  for (int e = threadIdx.x; e < r * r; e += blockDim.x) {
    md.M[e] = 0.f;
    md.Vm[e] = 0.f;
  }
}

}  // namespace

int32_t qr_block_rows(int32_t r) {
  switch (r) {
    case 4: return QrShape<4>::kB;
    case 8: return QrShape<8>::kB;
    case 16: return QrShape<16>::kB;
    case 32: return QrShape<32>::kB;
    case 64: return QrShape<64>::kB;
    case 128: return QrShape<128>::kB;
    default: return 0;
  }
}

cudaError_t launch_qr_up(const QrBlock* d_blocks, int32_t n_blocks, int32_t r, uint64_t seed,
                         uint32_t refresh_idx, uint32_t* /*d_status*/, cudaStream_t s) {
  if (n_blocks <= 0) return cudaSuccess;
  switch (r) {
    case 4: return launch_up_r<4>(d_blocks, n_blocks, seed, refresh_idx, s);
    case 8: return launch_up_r<8>(d_blocks, n_blocks, seed, refresh_idx, s);
    case 16: return launch_up_r<16>(d_blocks, n_blocks, seed, refresh_idx, s);
    case 32: return launch_up_r<32>(d_blocks, n_blocks, seed, refresh_idx, s);
    case 64: return launch_up_r<64>(d_blocks, n_blocks, seed, refresh_idx, s);
    case 128: return launch_up_r<128>(d_blocks, n_blocks, seed, refresh_idx, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_qr_down(const QrBlock* d_blocks, int32_t n_blocks, int32_t r,
                           uint32_t* /*d_status*/, cudaStream_t s) {
  if (n_blocks <= 0) return cudaSuccess;
  switch (r) {
    case 4: return launch_down_r<4>(d_blocks, n_blocks, s);
    case 8: return launch_down_r<8>(d_blocks, n_blocks, s);
    case 16: return launch_down_r<16>(d_blocks, n_blocks, s);
    case 32: return launch_down_r<32>(d_blocks, n_blocks, s);
    case 64: return launch_down_r<64>(d_blocks, n_blocks, s);
    case 128: return launch_down_r<128>(d_blocks, n_blocks, s);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_zero_moments(const MatDesc* d_mats, int32_t n_mats, int32_t r, cudaStream_t s) {
  if (n_mats <= 0) return cudaSuccess;
  zero_moments_kernel<<<n_mats, 256, 0, s>>>(d_mats, r);
  return cudaGetLastError();
}

}  // namespace zo
