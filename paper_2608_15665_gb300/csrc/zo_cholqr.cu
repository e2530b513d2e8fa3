// Subspace refresh for tall panels at r = 16 ... 128: Alg. 1's Haar factor by
// CholeskyQR2 (Fukaya, Nakatsukasa, Yanagisawa and Yamamoto, 2014).
//
// Alg. 1 wants Q of the QR factorisation of a Gaussian panel Omega (rows x r) with the
// signs fixed so that diag(R) > 0 (Eq. (11)).  That Q is unique, and it is also
// Omega R^-1 with R^T R = Omega^T Omega the Cholesky factorisation (whose diagonal is
// positive by construction).  One Cholesky QR in fp32 leaves Q orthogonal only to about
// kappa(Omega)^2 u; applied a second time to its own output it reaches O(u) when
// kappa(Omega)^2 u << 1 -- for a tall Gaussian panel (rows >= 4r), kappa <= ~3.  So per
// panel:
//   G1 = Omega^T Omega,  L1 L1^T = G1,  Q1 = Omega L1^-T,
//   G2 = Q1^T Q1,        L2 L2^T = G2,  Q  = Q1 L2^-T        (Q = Omega (L2^T L1^T)^-1),
// and Q lands in U (or V).  Every step but the two r x r Cholesky factorisations is a
// batched product over rows, so the refresh runs at the speed of those products instead
// of r dependent Householder steps per block.  Omega is drawn in the kernels from the
// counter contract (tags 2 / 3, element e = row * r + col at counter e / 4, lane e % 4),
// exactly as the TSQR of zo_qr.cu draws it; panels shorter than 4r keep the TSQR.
//
// Launches per refresh: gram(Omega, which also writes Omega to the panel), chol,
// apply(Omega -> Q1), gram(Q1), chol, apply(Q1 -> Q).  Every sum is one chain of fp32
// multiply-adds in a fixed order (a Gram element over the rows of a 1024-row chunk, then chunk by
// chunk; a factor's and a product's elements over their index), whatever the tiles: a refresh is
// bit-reproducible, whichever matrices share the context.  The tiles keep the chains because
// bf16 weights show them: with the rows of a chunk dealt to groups of threads (Q's error against
// 64 bits halves, 32B set 1.67 ms) a step of a 1 M-weight set moved by up to rel 1.3e-5.
//
// Bound: fp32 multiply-adds (8 r^2 per row over the four products, 5.3 r^2 with the triangles
// left out) and Omega's draws; at r = 128 on few panels the factorisations.  So: register tiles
// in packed multiply-adds, which shared memory can feed; only the Gram matrix's lower blocks;
// only L^-1's lower half where a thread's columns allow; Omega drawn once; and a blocked
// Cholesky.
// Refresh of 16 layers of the 32B set at r = 64: 2.64 -> 1.62 ms; of 32 of the 7B set at r = 32:
// 1.29 -> 0.88, of one 0.191 -> 0.132; of 8 at r = 128: 4.38 -> 1.82; of 24 of the 1.3B set at
// r = 16: 0.278 -> 0.182.
#include "zo_cluster.cuh"
#include "zo_fma_common.cuh"
#include "zo_kernels.h"
#include "zo_launch.cuh"

namespace zo {
namespace {

using namespace fma;

// ---------------------------------------------------------------- Gram matrices of chunks
// A CTA takes kG chunks; of each, T x T blocks of the lower triangle, a block per thread.  Every
// element is one chain of fp32 multiply-adds over the chunk's rows in order, whatever the tile,
// so tiles are free to follow the machine: 4 x 4 (2 x 2 at r = 16), because chains are what is
// short.  8 x 8 tiles load half as much from shared memory per multiply-add but leave a quarter
// of the warps: 1.91 ms for 16 layers of the 32B set at r = 64 where these take 1.70, 1.17
// against 0.89 for 32 of the 7B set at r = 32.  256 threads load or draw a stage even where fewer
// multiply (one 7B layer at r = 32, CTAs of the 64 that multiply: 205 us a refresh; of 256: 141).
// Rows pass through a ring of stages, copied two ahead or drawn one ahead.
//
// 4 layers of the 32B set at r = 64: 93 us, where the bytes take 20, the multiply-adds 34 and the
// shared-memory reads 69; Omega's draws add 63.
template <int R, int T, int kG, bool kOmega>
struct Gram {
  static constexpr int kN = R / T;
  static constexpr int kBlocks = kN * (kN + 1) / 2;
  static constexpr int kBlockThreads = (kBlocks * kG + 31) / 32 * 32;
  static constexpr int kThreads = kBlockThreads > 256 ? kBlockThreads : 256;
  static constexpr int kPer = 256 / kG;                               // loading threads of a chunk
  static constexpr int kSub = kG > 1 ? 32 : R == 16 ? 128 : R == 32 ? 64 : 32;
  static constexpr int kStages = kOmega ? 2 : 3;
  static constexpr int kLd = R + 4;
  static constexpr int kStage = kG * kSub * kLd;                      // floats
  static constexpr size_t kSmem = sizeof(float) * kStages * kStage;
  static_assert(kSub * R / 4 % kPer == 0, "whole words per loading thread");
};

// T consecutive floats as pairs
template <int T>
__device__ __forceinline__ void load_pairs(const float* p, float2 (&v)[T / 2]) {
  if constexpr (T == 2) {
    v[0] = *reinterpret_cast<const float2*>(p);
  } else {
#pragma unroll
    for (int q = 0; q < T / 4; ++q) {
      const float4 x = reinterpret_cast<const float4*>(p)[q];
      v[2 * q] = make_float2(x.x, x.y);
      v[2 * q + 1] = make_float2(x.z, x.w);
    }
  }
}

template <int R, int T, int kG, bool kOmega>
__global__ void __launch_bounds__(Gram<R, T, kG, kOmega>::kThreads)
cq_gram_kernel(const CqPanel* __restrict__ panels, const CqChunk* __restrict__ chunks, int n_chunks,
               float* __restrict__ partial, uint64_t seed, uint32_t refresh_idx) {
  using Cfg = Gram<R, T, kG, kOmega>;
  constexpr int kLd = Cfg::kLd, kW = R / 4, kStages = Cfg::kStages, kSub = Cfg::kSub, kP = T / 2;
  extern __shared__ __align__(16) float cq_smem[];
  __shared__ int rows[kG];
  const int tid = threadIdx.x, chunk0 = blockIdx.x * kG;
  // thread's chunk to load: 256 threads, kPer for each
  const int q = min(tid / Cfg::kPer, kG - 1), w0 = tid % Cfg::kPer;
  float* src = nullptr;                          // the chunk's rows in its panel
  int words = 0;                                 // 4-float words in them
  uint32_t c0 = 0, gidx = 0, tag = 0;            // the first one's counter; the stream
  if (tid < 256 && chunk0 + q < n_chunks) {
    const CqChunk ch = chunks[chunk0 + q];
    const CqPanel pn = panels[ch.panel];
    src = pn.out + ch.row0 * R;
    words = ch.nrows * kW;
    c0 = (uint32_t)((ch.row0 * R) >> 2);
    gidx = pn.gidx;
    tag = query_word(pn.tag, 0);
  }
  if (w0 == 0 && tid < 256) rows[q] = words / kW;
  if constexpr (kG == 1) {                       // the launches of few chunks are dependent
    pdl_wait();
    pdl_trigger();
  }
  __syncthreads();
  const int g = min(tid / Cfg::kBlocks, kG - 1), u = tid % Cfg::kBlocks;
  int bi = 0;
  while ((bi + 1) * (bi + 2) / 2 <= u) ++bi;
  const int bj = u - bi * (bi + 1) / 2;          // bj <= bi
  const bool mine = tid < Cfg::kBlocks * kG;
  int most = 0;
#pragma unroll
  for (int i = 0; i < kG; ++i) most = max(most, rows[i]);
  const int n_sub = (most + kSub - 1) / kSub;

  // stage t's rows: drawn (and kept in the panel), or copied
  auto stage = [&](int t) {
    if (t < n_sub) {
      float* dst = cq_smem + t % kStages * Cfg::kStage + q * kSub * kLd;
#pragma unroll
      for (int i = 0; i < kSub * kW / Cfg::kPer; ++i) {
        const int w = w0 + i * Cfg::kPer, v = t * kSub * kW + w;
        if (v >= words) continue;
        float* d = dst + w / kW * kLd + 4 * (w % kW);
        if constexpr (kOmega) {
          const float4 z = normal4(seed, c0 + (uint32_t)v, gidx, refresh_idx, tag);
          *reinterpret_cast<float4*>(src + 4 * v) = z;
          *reinterpret_cast<float4*>(d) = z;
        } else {
          cp_async_16(d, src + 4 * v, 16);
        }
      }
    }
    if constexpr (!kOmega) cp_async_commit();
  };

  // acc[e][a][b]: columns 2b, 2b + 1 of the block with rows 2a, 2a + 1 (e = 0) or 2a + 1, 2a
  // (e = 1): swapped pairs take half the register moves of duplicated operands
  float2 acc[2][kP][kP];
#pragma unroll
  for (int e = 0; e < 2 * kP * kP; ++e)
    acc[e / (kP * kP)][e / kP % kP][e % kP] = make_float2(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < kStages - 1; ++t) stage(t);
  for (int t = 0; t < n_sub; ++t) {
    if constexpr (!kOmega) cp_async_wait<kStages - 2>();
    __syncthreads();                             // stage t is there, stage t - 1 is read
    stage(t + kStages - 1);
    if (!mine) continue;
    const int n = min(kSub, rows[g] - t * kSub);
    const float* X = cq_smem + t % kStages * Cfg::kStage + g * kSub * kLd;
#pragma unroll 4
    for (int k = 0; k < n; ++k) {
      float2 a2[kP], b2[kP];
      load_pairs<T>(X + k * kLd + T * bi, a2);
      load_pairs<T>(X + k * kLd + T * bj, b2);
#pragma unroll
      for (int a = 0; a < kP; ++a) {
        const float2 sw = make_float2(a2[a].y, a2[a].x);
#pragma unroll
        for (int b = 0; b < kP; ++b) {
          acc[0][a][b] = fma2(a2[a], b2[b], acc[0][a][b]);
          acc[1][a][b] = fma2(sw, b2[b], acc[1][a][b]);
        }
      }
    }
  }
  if (!mine || rows[g] == 0) return;
  float* out = partial + (int64_t)(chunk0 + g) * R * R + T * bi * R + T * bj;
#pragma unroll
  for (int a = 0; a < kP; ++a)
#pragma unroll
    for (int b = 0; b < kP; ++b) {
      const float2 d = acc[0][a][b], x = acc[1][a][b];
      *reinterpret_cast<float2*>(out + 2 * a * R + 2 * b) = make_float2(d.x, x.y);
      *reinterpret_cast<float2*>(out + (2 * a + 1) * R + 2 * b) = make_float2(x.x, d.y);
    }
}

template <int R, int T, int kG, bool kOmega>
cudaError_t launch_gram(const CqPanel* d_panels, const CqChunk* d_chunks, int32_t n_chunks,
                        float* d_partial, uint64_t seed, uint32_t refresh_idx, bool dependent,
                        cudaStream_t s) {
  using Cfg = Gram<R, T, kG, kOmega>;
  const cudaError_t e = cudaFuncSetAttribute(
      cq_gram_kernel<R, T, kG, kOmega>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::kSmem);
  if (e != cudaSuccess) return e;
  return launch_dependent(cq_gram_kernel<R, T, kG, kOmega>, (unsigned)((n_chunks + kG - 1) / kG),
                          Cfg::kThreads, Cfg::kSmem, s, 1, dependent, d_panels, d_chunks, n_chunks,
                          d_partial, seed, refresh_idx);
}

// ---------------------------------------------------------------- Cholesky factor, inverse
// A cluster of CTAs per panel sums its chunk partials (chunk order, lower triangle; 50 of them
// at 25600 rows and r = 64), each CTA every fourth row of G, into the first CTA's shared
// memory.  The first goes on alone: G's Cholesky factor L (G = L L^T) and L^-1 in blocks of 16
// columns; it writes the transpose of L^-1 (zeros below the diagonal) to linv[panel].  A
// non-positive pivot -- not expected for a tall Gaussian panel -- sets kDevNotPosDef and leaves
// L^-1 = 0.
//
// Latency-bound: a block's columns are one warp's registers, so that the CTA synchronises 3
// times per 16 columns instead of 3 times per column, and the products around them, those of
// the inverse among them, run on all threads.  56 panels at r = 128: 440 -> 78 us; at r = 64:
// 113 -> 32 us (the inverse's divisions, part of its chains, are 10 of the 78).
constexpr int kCholCtas = 4;
constexpr int kNb = 16;
template <int R>
constexpr int kCholThreads = R == 128 ? 512 : 256;   // >= R: phase 2

template <int R>
__global__ void __launch_bounds__(kCholThreads<R>)
cq_chol_kernel(const CqPanel* __restrict__ panels, const float* __restrict__ partial,
               float* __restrict__ linv, uint32_t* __restrict__ status) {
  constexpr int kLd = R + 1, kBlks = R / kNb, kThreads = kCholThreads<R>;
  extern __shared__ float cq_smem[];
  // R x kLd: G, whose lower triangle becomes L below its diagonal blocks; the transpose of L^-1
  // (on the way, of the L L^-1 of rows to come) in the diagonal blocks and above
  float* A = cq_smem;
  __shared__ float LT[kNb][kNb], diag[kNb], dinv[kNb];   // LT[j][i] = L[k0 + i][k0 + j]
  __shared__ int bad;
  const CqPanel pn = panels[blockIdx.x / kCholCtas];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = blockIdx.x % kCholCtas;
  if (rank == 0) {
    for (int e = tid; e < R * R; e += kThreads)
      if (e % R > e / R) A[e / R * kLd + e % R] = 0.f;
    if (tid == 0) bad = 0;
  }
  cta2::cluster_sync_all();                      // all CTAs of the cluster run
  pdl_wait();
  pdl_trigger();
  const uint32_t a0 = cta2::map_to(A, 0);
  for (int w = tid; w < R * R / 4 / kCholCtas; w += kThreads) {
    const int i = w / (R / 4) * kCholCtas + rank, j = 4 * (w % (R / 4));
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    if (j > i) continue;
    const float4* p = reinterpret_cast<const float4*>(partial + (int64_t)pn.chunk0 * R * R + i * R + j);
#pragma unroll 8
    for (int c = 0; c < pn.n_chunks; ++c) {
      const float4 v = p[(int64_t)c * (R * R / 4)];
      s = make_float4(s.x + v.x, s.y + v.y, s.z + v.z, s.w + v.w);
    }
    const float v[4] = {s.x, s.y, s.z, s.w};
#pragma unroll
    for (int q = 0; q < 4; ++q)
      if (j + q <= i)
        asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a0 + 4u * (uint32_t)(i * kLd + j + q)),
                     "f"(v[q]) : "memory");
  }
  cta2::cluster_sync_all();                      // G is in the first CTA
  if (rank != 0) return;
  for (int kb = 0; kb < kBlks; ++kb) {
    const int k0 = kb * kNb;
    if (warp == 0) {
      // Phase 1: the diagonal block's factor, row k0 + lane
      float a[kNb];
      const int row = lane & (kNb - 1);
#pragma unroll
      for (int j = 0; j < kNb; ++j) a[j] = A[(k0 + row) * kLd + k0 + j];
      bool neg = false;
#pragma unroll
      for (int j = 0; j < kNb; ++j) {
        const float d = __shfl_sync(0xffffffffu, a[j], j);
        neg = neg || !(d > 0.f);
        const float l = sqrtf(d > 0.f ? d : 1.f), inv = 1.f / l;
        if (lane == j) {
          diag[j] = l;
          dinv[j] = inv;
        }
        a[j] = row == j ? l : a[j] * inv;
#pragma unroll
        for (int k = 0; k < kNb; ++k) {
          if (k <= j) continue;
          const float lk = __shfl_sync(0xffffffffu, a[j], k);
          if (row >= k) a[k] = fmaf(-a[j], lk, a[k]);
        }
      }
      if (lane < kNb)
#pragma unroll
        for (int j = 0; j < kNb; ++j) LT[j][row] = a[j];
      if (neg && lane == 0) bad = 1;
    }
    __syncthreads();
    // Phase 2, a thread each: a row below, L_21 (its 16 entries by substitution from the left);
    // or a column of L^-1's rows k0 .. (from what phase 3 has summed there, or the unit column).
    const int n_rows = R - k0 - kNb;
    if (tid < R) {
      const bool below = tid < n_rows;
      const int col = tid - n_rows;                        // of L^-1, < k0 + kNb
      float* p = A + (below ? k0 + kNb + tid : col) * kLd + k0;
      const int top = below ? -1 : col - k0;               // >= 0: the column's pivot row
      float x[kNb];
#pragma unroll
      for (int j = 0; j < kNb; ++j) x[j] = top >= 0 ? 0.f : p[j];
#pragma unroll
      for (int j = 0; j < kNb; ++j) {
        if (below) x[j] *= dinv[j];
        else if (j > top) x[j] = -x[j] / diag[j];
        else if (j == top) x[j] = dinv[j];
        const float m = below ? -x[j] : x[j];
#pragma unroll
        for (int k = 0; k < kNb; ++k)
          if (k > j) x[k] = fmaf(m, LT[j][k], x[k]);
      }
#pragma unroll
      for (int j = 0; j < kNb; ++j) p[j] = x[j];
    }
    __syncthreads();
    // Phase 3, in 4 x 4 tiles of rows nt apart (and columns nt or ct apart): G_22 -= L_21
    // L_21^T, lower triangle; and below row block k0 of L^-1, L_21 times it.
    const int nt = n_rows / 4, ct = (k0 + kNb) / 4;
    for (int w = tid; w < nt * (nt + ct); w += kThreads) {
      if (w < nt * nt) {
        float s[4][4];
        const int ti = w / nt, tj = w % nt;
        const float* x = A + (k0 + kNb + ti) * kLd + k0;
        const float* y = A + (k0 + kNb + tj) * kLd + k0;
        float* g = A + (k0 + kNb + ti) * kLd + k0 + kNb + tj;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < i || (j == i && tj <= ti)) s[i][j] = g[i * nt * kLd + j * nt];
#pragma unroll
        for (int k = 0; k < kNb; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j <= i) s[i][j] = fmaf(-x[i * nt * kLd + k], y[j * nt * kLd + k], s[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < i || (j == i && tj <= ti)) g[i * nt * kLd + j * nt] = s[i][j];
      } else {
        float s[4][4];
        const int ti = (w - nt * nt) / ct, tj = (w - nt * nt) % ct;
        const float* x = A + (k0 + kNb + ti) * kLd + k0;
        const float* y = A + tj * kLd + k0;
        float* g = A + tj * kLd + k0 + kNb + ti;
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) s[i][j] = g[j * ct * kLd + i * nt];
#pragma unroll
        for (int k = 0; k < kNb; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              s[i][j] = fmaf(x[i * nt * kLd + k], y[j * ct * kLd + k], s[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j) g[j * ct * kLd + i * nt] = s[i][j];
      }
    }
    __syncthreads();
  }
  float* out = linv + (int64_t)(blockIdx.x / kCholCtas) * R * R;
  for (int e = tid; e < R * R; e += kThreads)
    out[e] = bad || e % R / kNb < e / R / kNb ? 0.f : A[e / R * kLd + e % R];
  if (tid == 0 && bad) atomicOr(status, (uint32_t)kDevNotPosDef);
}

// ---------------------------------------------------------------- Q rows = X rows L^-T
// out[j][a] = sum_{b <= a} X[j][b] Linv[a][b] over one chunk, in place, in tiles of kRows rows:
// dealt to gridDim.y CTAs, X and Linv's transpose LT[b][a] row-major in shared memory.  Thread
// (ry, tx) owns rows ry + kRowThreads i and columns 4 tx .. + 3 of either half of the columns;
// past half of b only the second half's are left.  Several small CTAs per SM overlap one's copies
// with the others' multiply-adds (two of 256 threads on 256 rows: a refresh of 16 layers of the
// 32B set at r = 64 1.70 ms; four of 128 on 128 rows: 1.62).  Of about 70 us for 4 layers, 31
// are for the bytes, 44 for the multiply-adds and 49 for the shared-memory reads.
template <int R>
struct Apply {
  static constexpr int kThreads = R == 128 ? 256 : 128;
  static constexpr int kColThreads = R / 8;
  static constexpr int kRowThreads = kThreads / kColThreads;          // 64, 32, 16, 16
  static constexpr int kTR = R == 16 ? 2 : R == 64 ? 8 : 4;           // rows per thread
  static constexpr int kRows = kRowThreads * kTR;                     // 128; 64 at R = 128
  static constexpr int kLd = R + 4;
  static constexpr size_t kSmem = sizeof(float) * ((size_t)kRows + R) * kLd;
};

template <int R>
__global__ void __launch_bounds__(Apply<R>::kThreads, R <= 32 ? 6 : R == 64 ? 4 : 2)
cq_apply_kernel(const CqPanel* __restrict__ panels, const CqChunk* __restrict__ chunks,
                const float* __restrict__ linv) {
  using Cfg = Apply<R>;
  constexpr int kLd = Cfg::kLd, kW = R / 4, kTR = Cfg::kTR;
  extern __shared__ float cq_smem[];
  float* X = cq_smem;                            // kRows x kLd
  float* LT = cq_smem + Cfg::kRows * kLd;        // R x kLd
  const CqChunk ch = chunks[blockIdx.x];
  const CqPanel pn = panels[ch.panel];
  const int tid = threadIdx.x, tx = tid % Cfg::kColThreads, ry = tid / Cfg::kColThreads;
  const float* L = linv + (int64_t)ch.panel * R * R;
  pdl_wait();
  pdl_trigger();
  // a short chunk leaves CTAs without rows: they must not start copies that nothing waits for
  if ((int)blockIdx.y * Cfg::kRows >= ch.nrows) return;
  for (int w = tid; w < R * kW; w += Cfg::kThreads)
    cp_async_16(LT + (w / kW) * kLd + 4 * (w % kW), L + 4 * w, 16);
  for (int s0 = blockIdx.y * Cfg::kRows; s0 < ch.nrows; s0 += gridDim.y * Cfg::kRows) {
    const int n = min(Cfg::kRows, ch.nrows - s0);
    float* rows = pn.out + (ch.row0 + s0) * R;
    __syncthreads();
    for (int w = tid; w < n * kW; w += Cfg::kThreads)
      cp_async_16(X + (w / kW) * kLd + 4 * (w % kW), rows + 4 * (int64_t)w, 16);
    cp_async_commit();
    cp_async_wait<0>();
    __syncthreads();
    float2 acc[kTR][4];
#pragma unroll
    for (int i = 0; i < kTR; ++i)
#pragma unroll
      for (int c = 0; c < 4; ++c) acc[i][c] = make_float2(0.f, 0.f);
#pragma unroll
    for (int half = 0; half < 2; ++half) {
#pragma unroll 2
      for (int b4 = half * kW / 2; b4 < (half + 1) * kW / 2; ++b4) {
        float4 x[kTR];
#pragma unroll
        for (int i = 0; i < kTR; ++i)
          x[i] = *reinterpret_cast<const float4*>(X + (ry + Cfg::kRowThreads * i) * kLd + 4 * b4);
#pragma unroll
        for (int bb = 0; bb < 4; ++bb) {
          const float* l = LT + (4 * b4 + bb) * kLd + 4 * tx;
          const float4 l1 = *reinterpret_cast<const float4*>(l + R / 2);
          const float4 l0 = half == 0 ? *reinterpret_cast<const float4*>(l) : l1;
#pragma unroll
          for (int i = 0; i < kTR; ++i) {
            const float xv = bb == 0 ? x[i].x : bb == 1 ? x[i].y : bb == 2 ? x[i].z : x[i].w;
            const float2 x2 = make_float2(xv, xv);
            if (half == 0) {
              acc[i][0] = fma2(x2, make_float2(l0.x, l0.y), acc[i][0]);
              acc[i][1] = fma2(x2, make_float2(l0.z, l0.w), acc[i][1]);
            }
            acc[i][2] = fma2(x2, make_float2(l1.x, l1.y), acc[i][2]);
            acc[i][3] = fma2(x2, make_float2(l1.z, l1.w), acc[i][3]);
          }
        }
      }
    }
#pragma unroll
    for (int i = 0; i < kTR; ++i) {
      const int j = ry + Cfg::kRowThreads * i;
      if (j >= n) continue;
      float* q = rows + (int64_t)j * R + 4 * tx;
      *reinterpret_cast<float4*>(q) = make_float4(acc[i][0].x, acc[i][0].y, acc[i][1].x, acc[i][1].y);
      *reinterpret_cast<float4*>(q + R / 2) =
          make_float4(acc[i][2].x, acc[i][2].y, acc[i][3].x, acc[i][3].y);
    }
  }
}

template <int R>
size_t chol_smem() { return sizeof(float) * R * (R + 1); }

template <int R>
cudaError_t run_cholqr_r(const CqPanel* d_panels, int32_t n_panels, const CqChunk* d_chunks,
                         int32_t n_chunks, float* d_partial, float* d_linv, uint64_t seed,
                         uint32_t refresh_idx, int32_t sms, uint32_t* d_status, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(cq_chol_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)chol_smem<R>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cq_apply_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Apply<R>::kSmem);
  if (e != cudaSuccess) return e;
  constexpr int kT = R == 16 ? 2 : 4, kG = R == 128 ? 1 : 2;
  // Fewer than four chunks per SM: a CTA of the Gram kernels each, and launches that wait for
  // their predecessor and overlap its tail; else kG chunks per CTA and ordinary launches.  A
  // refresh in us on 152 SMs, this way / the other, of 4096 x 1024 matrices:
  //   chunks     80       320        610        960         1280         2560         3840
  //   r = 16   67 / 111  104 / 132  143 / 165  193 / 214   253 / 268    471 / 490    687 / 677
  //   r = 32  133 / 157  206 / 219  300 / 314  443 / 432   541 / 539    989 / 962   1472 / 1385
  //   r = 64  194 / 266  376 / 458  634 / 686  899 / 957  1126 / 1196  2117 / 2172  3153 / 3139
  // (whole layers of the 1.3B, 7B and 32B sets alike).  The line is r = 32's; at r = 16 and 64,
  // where it leaves 2 to 15% between 608 and some 2500 chunks, it is kept for one rule.
  const bool few = n_chunks < 4 * sms;
  // Not dependent at r = 128, where the next kernel's large CTAs take the SM from this one's (one
  // 7B layer: 467 -> 512 us).
  const bool dep = few && R < 128;
  // CTAs per chunk of the triangular product.  r < 128: eight, a 128-row tile each.  r = 128: two
  // 64-row tiles each, four where chunks are many, for the 64 KB of L^-1 that each CTA copies
  // (4096 x 1024 matrices, eight / four CTAs: 469 / 488 us at 80 chunks, 1187 / 1188 at 320, 1658 /
  // 1636 at 480, 2022 / 2005 at 610, 3839 / 3755 at 1280).
  const int n_split = R < 128 || few ? 8 : 4;
  // first Cholesky QR: Omega -> Q1; second: Q1 -> Q; both in the panels
  for (int round = 0; round < 2; ++round) {
    if (few)
      e = round == 0 ? launch_gram<R, kT, 1, true>(d_panels, d_chunks, n_chunks, d_partial, seed, refresh_idx, dep, s)
                     : launch_gram<R, kT, 1, false>(d_panels, d_chunks, n_chunks, d_partial, seed, refresh_idx, dep, s);
    else
      e = round == 0 ? launch_gram<R, kT, kG, true>(d_panels, d_chunks, n_chunks, d_partial, seed, refresh_idx, dep, s)
                     : launch_gram<R, kT, kG, false>(d_panels, d_chunks, n_chunks, d_partial, seed, refresh_idx, dep, s);
    if (e != cudaSuccess) return e;
    e = launch_dependent(cq_chol_kernel<R>, (unsigned)(n_panels * kCholCtas), kCholThreads<R>,
                         chol_smem<R>(), s, kCholCtas, dep, d_panels, d_partial, d_linv, d_status);
    if (e != cudaSuccess) return e;
    e = launch_dependent(cq_apply_kernel<R>, dim3(n_chunks, n_split), Apply<R>::kThreads,
                         Apply<R>::kSmem, s, 1, dep, d_panels, d_chunks, d_linv);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

bool cholqr_supported(int32_t r) { return r == 16 || r == 32 || r == 64 || r == 128; }

cudaError_t launch_cholqr(const CqPanel* d_panels, int32_t n_panels, const CqChunk* d_chunks,
                          int32_t n_chunks, float* d_partial, float* d_linv, int32_t r,
                          uint64_t seed, uint32_t refresh_idx, int32_t sms, uint32_t* d_status,
                          cudaStream_t s) {
  if (n_panels <= 0) return cudaSuccess;
  switch (r) {
    case 16: return run_cholqr_r<16>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, sms, d_status, s);
    case 32: return run_cholqr_r<32>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, sms, d_status, s);
    case 64: return run_cholqr_r<64>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, sms, d_status, s);
    case 128: return run_cholqr_r<128>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, sms, d_status, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zo
