// Per-pass r x r coefficient C_i and its projection P_i = C_i V_i^T.
//
// Every weight pass of the library has the form W_i <- rnd(W_i + U_i C_i V_i^T)
// (Alg. 2 / Eq. (4), with consecutive updates fused).  C_i is formed here, one
// CTA per matrix, from the Gaussian Z_i^(k) of the counter contract:
//   perturb: C_i = eps (ca Z_i^(qa) + cb Z_i^(qb))
//   step:    rho_k from the losses (Eq. (3) central / Eq. (6) forward),
//            G_i = (1/q) sum_k rho_k Z_i^(k)                       (Eq. (6), Alg. 3)
//            Adam: M <- b1 M + (1-b1) G, Vm <- b2 Vm + (1-b2) G.G  (Eqs. (7), (8))
//                  D = (M / (1-b1^t)) / (sqrt(Vm / (1-b2^t)) + eps_adam)  (Eqs. (9), (10))
//            SGD:  D = G                                              (Sec. 3)
//            C_i = -lr D + restore_coef eps Z_i^(restore_query)
// P_i = C_i V_i^T (r x n) then feeds the weight pass.  For the tensor-core path the kernel
// also writes C_i as the projection's operand, rows [hi | lo] of the fp16 pair of
// C_i 2^(e_C,i) with e_C,i from max |C_i| (zo_tc_common.cuh), and pinv_i = 2^-(e_P,i).
//
// One CTA per matrix up to r = 32, a cluster of four at r = 64 and of eight at r = 128 (the
// maximum and the norm meet through distributed shared memory): at most two counters per
// thread.  Latency-bound: the perturbation's draws, which need no memory, come before the
// wait for the stream's previous kernel.
#include "zo_cluster.cuh"
#include "zo_kernels.h"
#include "zo_launch.cuh"
#include "zo_tc_common.cuh"

namespace zo {
namespace {

constexpr int kMaxQ = 4096;

__device__ __forceinline__ float4 f4_axpy(float a, float4 x, float4 y) {  // a*x + y
  return make_float4(fmaf(a, x.x, y.x), fmaf(a, x.y, y.y), fmaf(a, x.z, y.z), fmaf(a, x.w, y.w));
}
__device__ __forceinline__ float4 f4_scale(float a, float4 x) {
  return make_float4(a * x.x, a * x.y, a * x.z, a * x.w);
}

constexpr int kCoeffThreads = 256;
constexpr int kCoeffIters = 2;              // counters per thread
__host__ __device__ constexpr int coeff_ctas(int r) { return r == 128 ? 8 : r == 64 ? 4 : 1; }

__global__ void __launch_bounds__(kCoeffThreads)
coeff_kernel(const MatDesc* __restrict__ mats, const CoeffParams p) {
  extern __shared__ float rho_s[];          // q values (step mode)
  __shared__ float sum_s[8], max_s[8];
  __shared__ float cta_sum, cta_max;
  const int r = p.r, ctas = coeff_ctas(r);
  const int i = (int)(blockIdx.x / ctas), rank = (int)(blockIdx.x % ctas);
  const MatDesc md = mats[i];
  const int n_ctr = r * r / 4;              // r is a multiple of 4, so r * r of 16
  const int per = n_ctr / ctas;             // this CTA's counters
  const int c0 = rank * per;
  const int tid = threadIdx.x;
  float4 out[kCoeffIters];

  if (p.mode == kCoeffPerturb) {
#pragma unroll
    for (int k = 0; k < kCoeffIters; ++k) {
      const int c = tid + k * kCoeffThreads;
      if (c >= per) break;
      float4 acc = f4_scale(p.ca, normal4(p.seed, (uint32_t)(c0 + c), md.gidx, p.t,
                                          query_word(kTagZ, (uint32_t)p.qa)));
      if (p.qb >= 0)
        acc = f4_axpy(p.cb, normal4(p.seed, (uint32_t)(c0 + c), md.gidx, p.t,
                                    query_word(kTagZ, (uint32_t)p.qb)), acc);
      out[k] = f4_scale(p.eps, acc);
    }
  }
  pdl_wait();
  pdl_trigger();

  float gsq = 0.0f;
  if (p.mode == kCoeffStep) {
    for (int k = tid; k < p.q; k += kCoeffThreads) {
      float rho;
      if (p.scheme == 0) {          // central: (L+_k - L-_k) / (2 eps)
        rho = (p.losses[2 * k] - p.losses[2 * k + 1]) / (2.0f * p.eps);
      } else if (p.scheme == 1) {   // forward: (l_(k+1) - l_0) / eps
        rho = (p.losses[k + 1] - p.losses[0]) / p.eps;
      } else {                      // rho given directly
        rho = p.losses[k];
      }
      rho_s[k] = rho;
    }
    __syncthreads();
#pragma unroll
    for (int it = 0; it < kCoeffIters; ++it) {
      if (tid + it * kCoeffThreads >= per) break;
      const int c = c0 + tid + it * kCoeffThreads;
      // G: accumulate in query order, then divide by q (Alg. 3)
      float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int k = 0; k < p.q; ++k)
        g = f4_axpy(rho_s[k], normal4(p.seed, (uint32_t)c, md.gidx, p.t,
                                      query_word(kTagZ, (uint32_t)k)), g);
      const float fq = (float)p.q;
      g = make_float4(g.x / fq, g.y / fq, g.z / fq, g.w / fq);
      gsq += g.x * g.x + g.y * g.y + g.z * g.z + g.w * g.w;
      float4 d;
      if (p.optimizer == 0) {
        float4* M4 = reinterpret_cast<float4*>(md.M);
        float4* V4 = reinterpret_cast<float4*>(md.Vm);
        float4 m = M4[c], v = V4[c];
        const float b1 = p.beta1, b2 = p.beta2;
        const float a1 = 1.0f - b1, a2 = 1.0f - b2;
        m = make_float4(b1 * m.x + a1 * g.x, b1 * m.y + a1 * g.y, b1 * m.z + a1 * g.z,
                        b1 * m.w + a1 * g.w);
        v = make_float4(b2 * v.x + a2 * (g.x * g.x), b2 * v.y + a2 * (g.y * g.y),
                        b2 * v.z + a2 * (g.z * g.z), b2 * v.w + a2 * (g.w * g.w));
        M4[c] = m;
        V4[c] = v;
        d.x = (m.x * p.inv_bc1) / (sqrtf(v.x * p.inv_bc2) + p.eps_adam);
        d.y = (m.y * p.inv_bc1) / (sqrtf(v.y * p.inv_bc2) + p.eps_adam);
        d.z = (m.z * p.inv_bc1) / (sqrtf(v.z * p.inv_bc2) + p.eps_adam);
        d.w = (m.w * p.inv_bc1) / (sqrtf(v.w * p.inv_bc2) + p.eps_adam);
      } else {
        d = g;
      }
      out[it] = f4_scale(-p.lr, d);
      if (p.restore_query >= 0) {
        const float4 z = normal4(p.seed, (uint32_t)c, md.gidx, p.t,
                                 query_word(kTagZ, (uint32_t)p.restore_query));
        out[it] = f4_axpy(p.restore_coef * p.eps, z, out[it]);
      }
    }
  }

  float cmax = 0.0f;
#pragma unroll
  for (int it = 0; it < kCoeffIters; ++it) {
    if (tid + it * kCoeffThreads >= per) break;
    const float4 o = out[it];
    reinterpret_cast<float4*>(md.C)[c0 + tid + it * kCoeffThreads] = o;
    cmax = fmaxf(cmax, fmaxf(fmaxf(fabsf(o.x), fabsf(o.y)), fmaxf(fabsf(o.z), fabsf(o.w))));
  }
  const bool gamma = p.mode == kCoeffStep && p.gamma_out != nullptr;
  if (p.c_hl == nullptr && !gamma) return;

  // max |C_i| and sum G_i^2 over the CTA, then (in rank order) the cluster
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    cmax = fmaxf(cmax, __shfl_xor_sync(0xffffffffu, cmax, o));
    gsq += __shfl_xor_sync(0xffffffffu, gsq, o);
  }
  if ((tid & 31) == 0) {
    max_s[tid >> 5] = cmax;
    sum_s[tid >> 5] = gsq;
  }
  __syncthreads();
  cmax = gsq = 0.f;
#pragma unroll
  for (int w = 0; w < kCoeffThreads / 32; ++w) {
    cmax = fmaxf(cmax, max_s[w]);
    gsq += sum_s[w];
  }
  if (ctas > 1) {
    if (tid == 0) {
      cta_max = cmax;
      cta_sum = gsq;
    }
    cta2::cluster_sync_all();
    cmax = gsq = 0.f;
    for (int c = 0; c < ctas; ++c) {
      float m, g;
      asm volatile("ld.shared::cluster.f32 %0, [%1];"
                   : "=f"(m) : "r"(cta2::map_to(&cta_max, (uint32_t)c)) : "memory");
      asm volatile("ld.shared::cluster.f32 %0, [%1];"
                   : "=f"(g) : "r"(cta2::map_to(&cta_sum, (uint32_t)c)) : "memory");
      cmax = fmaxf(cmax, m);
      gsq += g;
    }
  }
  if (gamma && rank == 0 && tid == 0) p.gamma_out[i] = sqrtf(gsq);
  if (p.c_hl != nullptr) {
    const int e_c = tc::coeff_scale_exp(cmax);
    if (rank == 0 && tid == 0) p.pinv[i] = tc::exp2i(-(e_c + tc::p_scale_offset(r)));
    const float scale = tc::exp2i(e_c);
    const int width = tc::hl_width(r);
#pragma unroll
    for (int it = 0; it < kCoeffIters; ++it) {
      if (tid + it * kCoeffThreads >= per) break;
      const int e = 4 * (c0 + tid + it * kCoeffThreads);
      uint2 hi, lo;
      tc::split4_f16(out[it], scale, hi, lo);
      uint16_t* row = p.c_hl + ((int64_t)i * r + e / r) * width + e % r;
      *reinterpret_cast<uint2*>(row) = hi;
      *reinterpret_cast<uint2*>(row + r) = lo;
    }
  }
  if (ctas > 1) cta2::cluster_sync_all();   // the peers have read this CTA's values
}

// P[a][j] = sum_b C[a][b] V[j][b], r = 4 and 8; one thread per column j, rows a split over ty.
template <int R>
__global__ void __launch_bounds__(256) project_fma_kernel(const MatDesc* __restrict__ mats,
                                                          const int2* __restrict__ units) {
  extern __shared__ float Cs[];   // R x R
  const int2 u = units[blockIdx.x];
  const MatDesc md = mats[u.x];
  const int tid = threadIdx.x;
  pdl_wait();
  pdl_trigger();
  for (int e = tid; e < R * R; e += blockDim.x) Cs[e] = md.C[e];
  __syncthreads();
  const int64_t j = (int64_t)u.y + (tid & 127);
  if (j >= md.n) return;
  float v[R];
  const float4* vrow = reinterpret_cast<const float4*>(md.V + j * R);
#pragma unroll
  for (int b = 0; b < R / 4; ++b) {
    const float4 t = vrow[b];
    v[4 * b] = t.x; v[4 * b + 1] = t.y; v[4 * b + 2] = t.z; v[4 * b + 3] = t.w;
  }
  for (int a = tid >> 7; a < R; a += 2) {
    const float4* crow = reinterpret_cast<const float4*>(Cs + a * R);
    float acc = 0.f;
#pragma unroll
    for (int b4 = 0; b4 < R / 4; ++b4) {
      const float4 c4 = crow[b4];
      acc = fmaf(c4.x, v[4 * b4], acc);
      acc = fmaf(c4.y, v[4 * b4 + 1], acc);
      acc = fmaf(c4.z, v[4 * b4 + 2], acc);
      acc = fmaf(c4.w, v[4 * b4 + 3], acc);
    }
    md.P[(int64_t)a * md.n + j] = acc;
  }
}

// The same at r = 16 ... 128 (the same terms in the same order): 128 columns by kRows rows of P
// per CTA, a warp's lanes the columns j, j + 32, j + 64, j + 96 and its kTR rows, so that four
// words of V and a quarter of a row's C feed 4 kTR multiply-adds (packed in pairs of columns).
// Bound by shared-memory reads; the thread-per-column form read 16 bytes of C for 4 of them and
// kept V's row in registers (r = 128: spilled to local memory).  V's 128 rows are transposed
// into shared memory with an odd pitch, by 16-byte loads of eight lanes to a row, before the
// wait: the coefficient kernel, always the stream's previous launch, triggers this one only
// after all work before it has completed, and writes no V.
// 12 layers of 768-wide matrices (83 K columns), the passes beside their weight kernels: 11.3 ->
// 5.5 us at r = 32, 39 -> 24 at r = 64, 182 -> 82 at r = 128.
template <int R>
struct ProjectTile {
  static constexpr int kRows = R < 64 ? R : 64;
  static constexpr int kTR = kRows / 8;               // rows of a warp: 2, 4, 8, 8
  static constexpr int kSplit = R / kRows;
  static constexpr int kCols = 128, kLd = kCols + 1;
  static constexpr size_t kSmem = sizeof(float) * (kRows * R + R * kLd);
};

template <int R>
__global__ void __launch_bounds__(256) project_tile_kernel(const MatDesc* __restrict__ mats,
                                                           const int2* __restrict__ units) {
  using T = ProjectTile<R>;
  constexpr int kLd = T::kLd, kTR = T::kTR, kCk = R < 32 ? R : 32;   // columns of V per sweep
  extern __shared__ float4 smem4[];
  float* Cs = reinterpret_cast<float*>(smem4);        // kRows x R
  float* Vs = Cs + T::kRows * R;                      // R x kLd
  const int2 u = units[blockIdx.x / T::kSplit];
  const int a0 = blockIdx.x % T::kSplit * T::kRows;
  const MatDesc md = mats[u.x];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
#pragma unroll 4
  for (int w = tid; w < T::kCols * R / 4; w += 256) {
    constexpr int kQ = kCk / 4;
    const int k = w / (T::kCols * kQ) * kCk + 4 * (w % kQ), j = w / kQ % T::kCols;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (u.y + j < md.n) v = *reinterpret_cast<const float4*>(md.V + ((int64_t)u.y + j) * R + k);
    float* d = Vs + k * kLd + j;
    d[0] = v.x; d[kLd] = v.y; d[2 * kLd] = v.z; d[3 * kLd] = v.w;
  }
  pdl_wait();
  pdl_trigger();
  const float4* C4 = reinterpret_cast<const float4*>(md.C + a0 * R);
  for (int e = tid; e < T::kRows * R / 4; e += 256) smem4[e] = C4[e];
  __syncthreads();
  float2 acc[kTR][2];
#pragma unroll
  for (int i = 0; i < kTR; ++i) acc[i][0] = acc[i][1] = make_float2(0.f, 0.f);
  const float* c = Cs + warp * kTR * R;
#pragma unroll 2
  for (int k4 = 0; k4 < R; k4 += 4) {
    float4 cv[kTR];
#pragma unroll
    for (int i = 0; i < kTR; ++i) cv[i] = *reinterpret_cast<const float4*>(c + i * R + k4);
#pragma unroll
    for (int kk = 0; kk < 4; ++kk) {
      const float* v = Vs + (k4 + kk) * kLd + lane;
      const float2 v0 = make_float2(v[0], v[32]), v1 = make_float2(v[64], v[96]);
#pragma unroll
      for (int i = 0; i < kTR; ++i) {
        const float x = kk == 0 ? cv[i].x : kk == 1 ? cv[i].y : kk == 2 ? cv[i].z : cv[i].w;
        acc[i][0] = fma2(make_float2(x, x), v0, acc[i][0]);
        acc[i][1] = fma2(make_float2(x, x), v1, acc[i][1]);
      }
    }
  }
  const int64_t j = (int64_t)u.y + lane;
#pragma unroll
  for (int i = 0; i < kTR; ++i) {
    float* p = md.P + (int64_t)(a0 + warp * kTR + i) * md.n;
    if (j < md.n) p[j] = acc[i][0].x;
    if (j + 32 < md.n) p[j + 32] = acc[i][0].y;
    if (j + 64 < md.n) p[j + 64] = acc[i][1].x;
    if (j + 96 < md.n) p[j + 96] = acc[i][1].y;
  }
}

template <int R>
cudaError_t launch_project_fma_r(const MatDesc* d_mats, const int2* d_units, int32_t n_units,
                                 cudaStream_t s) {
  if constexpr (R >= 16) {
    using T = ProjectTile<R>;
    const cudaError_t e = cudaFuncSetAttribute(
        project_tile_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)T::kSmem);
    if (e != cudaSuccess) return e;
    return launch_dependent(project_tile_kernel<R>, (unsigned)n_units * T::kSplit, 256, T::kSmem,
                            s, 1, true, d_mats, d_units);
  } else {
    return launch_dependent(project_fma_kernel<R>, (unsigned)n_units, 256, sizeof(float) * R * R, s,
                            1, true, d_mats, d_units);
  }
}

}  // namespace

cudaError_t launch_coeff(const MatDesc* d_mats, int32_t n_mats, const CoeffParams& p,
                         bool dependent, cudaStream_t s) {
  if (n_mats <= 0) return cudaSuccess;
  if (p.q > kMaxQ) return cudaErrorInvalidValue;
  const unsigned ctas = (unsigned)coeff_ctas(p.r);
  const size_t smem = p.mode == kCoeffStep ? sizeof(float) * p.q : 0;
  return launch_dependent(coeff_kernel, (unsigned)n_mats * ctas, kCoeffThreads, smem, s, ctas,
                          dependent, d_mats, p);
}

cudaError_t launch_project_fma(const MatDesc* d_mats, const int2* d_units, int32_t n_units,
                               int32_t r, cudaStream_t s) {
  if (n_units <= 0) return cudaSuccess;
  switch (r) {
    case 4: return launch_project_fma_r<4>(d_mats, d_units, n_units, s);
    case 8: return launch_project_fma_r<8>(d_mats, d_units, n_units, s);
    case 16: return launch_project_fma_r<16>(d_mats, d_units, n_units, s);
    case 32: return launch_project_fma_r<32>(d_mats, d_units, n_units, s);
    case 64: return launch_project_fma_r<64>(d_mats, d_units, n_units, s);
    case 128: return launch_project_fma_r<128>(d_mats, d_units, n_units, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zo
