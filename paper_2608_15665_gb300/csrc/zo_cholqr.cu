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
// apply(Omega -> Q1), gram(Q1), chol, apply(Q1 -> Q).  Sums over rows are fixed-order (groups
// of threads within a chunk of rows, then chunk by chunk), so a refresh is bit-reproducible.
//
// Bound: fp32 multiply-adds (8 r^2 per row over the four products, 5.3 r^2 with the triangles
// left out) and Omega's draws; at r = 128 on few panels the factorisations.  So: 8 x 8 (Gram)
// and up to 8 x 8 (apply) register tiles in packed multiply-adds, which shared memory can
// feed; only the Gram matrix's lower 8 x 8 blocks, the rows of a chunk dealt to as many groups
// of threads as the blocks leave room for; only L^-1's lower half where a thread's columns
// allow; Omega drawn once; and a blocked Cholesky.
// Refresh of 16 layers of the 32B set at r = 64: 2.64 -> 1.67 ms; of 32 of the 7B set at r = 32:
// 1.29 -> 0.81; of one at r = 128: 1.55 -> 0.44.  Q's error against 64 bits is 0.4 to 0.7 of
// the former kernels' (shorter chains of sums).
#include "zo_cluster.cuh"
#include "zo_fma_common.cuh"
#include "zo_kernels.h"
#include "zo_launch.cuh"

namespace zo {
namespace {

using namespace fma;

// ---------------------------------------------------------------- Gram matrix of a chunk
// 8 x 8 blocks of the lower triangle, a block of kGroups threads, which take the chunk's rows
// in turn.  Lanes of a warp read neighbouring rows of the same columns: with a row pitch of
// R + 4 floats no two of a load's 16-byte words share banks.  Rows pass through a ring of
// stages, copied two ahead (one ahead left the copies' latency exposed) or drawn one ahead.
// Bound by shared-memory reads and multiply-adds together: 4 16-byte loads per 32 packed
// multiply-adds, either 34 us of the 75 that 4 layers of the 32B set take at r = 64 (the bytes:
// 20); on Omega by its draws (another 59 us).
template <int R, bool kOmega>
struct Gram {
  static constexpr int kBlocks = (R / 8) * (R / 8 + 1) / 2;           // 3, 10, 36, 136
  static constexpr int kGroups = R == 16 ? 96 : R == 32 ? 32 : R == 64 ? 8 : 2;
  static constexpr int kThreads = (kBlocks * kGroups + 31) / 32 * 32;           // 288; 320 at R = 32
  static constexpr int kSub = R == 16 ? 384 : R == 32 ? 192 : R == 64 ? 64 : 32;   // rows of a stage
  static constexpr int kStages = kOmega ? 2 : 3;
  static constexpr int kLd = R + 4;
  static constexpr int kStage = kSub * kLd;                           // floats
  static constexpr size_t kSmem = sizeof(float) * kStages * kStage;
};

template <int R, bool kOmega>
__global__ void __launch_bounds__(Gram<R, kOmega>::kThreads, 2)
cq_gram_kernel(const CqPanel* __restrict__ panels, const CqChunk* __restrict__ chunks,
               float* __restrict__ partial, uint64_t seed, uint32_t refresh_idx) {
  using Cfg = Gram<R, kOmega>;
  constexpr int kLd = Cfg::kLd, kW = R / 4, kG = Cfg::kGroups, kStages = Cfg::kStages;
  extern __shared__ __align__(16) float cq_smem[];
  const CqChunk ch = chunks[blockIdx.x];
  const CqPanel pn = panels[ch.panel];
  const int tid = threadIdx.x, lane = tid & 31;
  const int g = tid % kG, u = min(tid / kG, Cfg::kBlocks - 1);
  int bi = 0;
  while ((bi + 1) * (bi + 2) / 2 <= u) ++bi;
  const int bj = u - bi * (bi + 1) / 2;                               // bj <= bi
  const int n_sub = (ch.nrows + Cfg::kSub - 1) / Cfg::kSub;

  // stage t's rows: drawn (and kept in the panel), or copied
  auto stage = [&](int t) {
    if (t < n_sub) {
      const int s0 = t * Cfg::kSub, n = min(Cfg::kSub, ch.nrows - s0);
      float* dst = cq_smem + t % kStages * Cfg::kStage;
      float* src = pn.out + (ch.row0 + s0) * R;
      for (int w = tid; w < n * kW; w += Cfg::kThreads) {
        float* d = dst + w / kW * kLd + 4 * (w % kW);
        if constexpr (kOmega) {
          const uint32_t c = (uint32_t)((((ch.row0 + s0) * R) >> 2) + w);
          const float4 z = normal4(seed, c, pn.gidx, refresh_idx, query_word(pn.tag, 0));
          *reinterpret_cast<float4*>(src + 4 * w) = z;
          *reinterpret_cast<float4*>(d) = z;
        } else {
          cp_async_16(d, src + 4 * w, 16);
        }
      }
    }
    if constexpr (!kOmega) cp_async_commit();
  };

  // acc[e][a][b]: columns 2b, 2b + 1 of the block with rows 2a, 2a + 1 (e = 0) or 2a + 1, 2a
  // (e = 1): swapped pairs take half the register moves of duplicated operands
  float2 acc[2][4][4];
#pragma unroll
  for (int e = 0; e < 32; ++e) acc[e / 16][e / 4 % 4][e % 4] = make_float2(0.f, 0.f);
#pragma unroll
  for (int t = 0; t < kStages - 1; ++t) stage(t);
  for (int t = 0; t < n_sub; ++t) {
    if constexpr (!kOmega) cp_async_wait<kStages - 2>();
    __syncthreads();                             // stage t is there, stage t - 1 is read
    stage(t + kStages - 1);
    const int n = min(Cfg::kSub, ch.nrows - t * Cfg::kSub);
    const float* X = cq_smem + t % kStages * Cfg::kStage;
#pragma unroll 2
    for (int k = g; k < n; k += kG) {
      const float4* xi = reinterpret_cast<const float4*>(X + k * kLd + 8 * bi);
      const float4* xj = reinterpret_cast<const float4*>(X + k * kLd + 8 * bj);
      const float4 i0 = xi[0], i1 = xi[1], j0 = xj[0], j1 = xj[1];
      const float2 a4[4] = {make_float2(i0.x, i0.y), make_float2(i0.z, i0.w),
                            make_float2(i1.x, i1.y), make_float2(i1.z, i1.w)};
      const float2 b4[4] = {make_float2(j0.x, j0.y), make_float2(j0.z, j0.w),
                            make_float2(j1.x, j1.y), make_float2(j1.z, j1.w)};
#pragma unroll
      for (int a = 0; a < 4; ++a) {
        const float2 sw = make_float2(a4[a].y, a4[a].x);
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          acc[0][a][b] = fma2(a4[a], b4[b], acc[0][a][b]);
          acc[1][a][b] = fma2(sw, b4[b], acc[1][a][b]);
        }
      }
    }
  }
  // The groups' sums, by halves: a lane hands the other half of its elements to its partner and
  // adds the partner's to its own, so it ends with the kKeep elements from kKeep (lane % kW2).
  constexpr int kW2 = kG < 32 ? kG : 32, kKeep = 64 / kW2;
  float v[64];
#pragma unroll
  for (int e = 0; e < 16; ++e) {
    const int a = e / 4, b = e % 4;
    v[16 * a + 2 * b] = acc[0][a][b].x;
    v[16 * a + 2 * b + 1] = acc[1][a][b].y;
    v[16 * a + 8 + 2 * b] = acc[1][a][b].x;
    v[16 * a + 8 + 2 * b + 1] = acc[0][a][b].y;
  }
#pragma unroll
  for (int off = kW2 / 2; off > 0; off /= 2) {
    const int n = off * kKeep;
    const bool up = lane & off;
#pragma unroll
    for (int i = 0; i < n; ++i) {
      const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
    }
  }
  const int m = kKeep * (lane % kW2);
  if constexpr (kG > 32) {                       // R = 16: a block is three warps' (kKeep = 2)
    __syncthreads();
    const int warp = tid / 32;
    if (warp % 3 > 0) *reinterpret_cast<float2*>(cq_smem + 64 * warp + m) = make_float2(v[0], v[1]);
    __syncthreads();
    if (warp % 3 > 0) return;
#pragma unroll
    for (int q = 1; q < 3; ++q) {
      const float2 o = *reinterpret_cast<const float2*>(cq_smem + 64 * (warp + q) + m);
      v[0] += o.x;
      v[1] += o.y;
    }
  }
  if (tid / kG >= Cfg::kBlocks) return;
  float* out = partial + (int64_t)blockIdx.x * R * R + (8 * bi + m / 8) * R + 8 * bj + m % 8;
  if constexpr (kKeep == 2) {
    *reinterpret_cast<float2*>(out) = make_float2(v[0], v[1]);
  } else {
#pragma unroll
    for (int q = 0; q < kKeep; q += 4)
      *reinterpret_cast<float4*>(out + q / 8 * R + q % 8) = make_float4(v[q], v[q + 1], v[q + 2], v[q + 3]);
  }
}

// ---------------------------------------------------------------- Cholesky factor, inverse
// A cluster of CTAs per panel sums its chunk partials (chunk order, lower triangle; 50 of them
// at 25600 rows and r = 64), each CTA every fourth row of G, into the first CTA's shared
// memory.  The first goes on alone: G's Cholesky factor L (G = L L^T) and L^-1 in blocks of 16
// columns; it writes the transpose of L^-1 (zeros below the diagonal) to linv[panel].  A
// non-positive pivot -- not expected for a tall Gaussian panel -- sets kDevNotPosDef and leaves
// L^-1 = 0.
//
// Latency-bound: a block's columns are one warp's registers, so that the CTA synchronises 4
// times per 16 columns instead of 3 times per column, and the products around them, those of
// the inverse among them, run on all threads.  56 panels at r = 128: 440 -> 64 us; at r = 64:
// 113 -> 28 us.  (One CTA per panel: 106 and 52.)
constexpr int kCholCtas = 4;
constexpr int kNb = 16;
template <int R>
constexpr int kCholThreads = R == 128 ? 512 : 256;   // >= 4 (R - kNb): phase 2, one item each

template <int R>
__global__ void __launch_bounds__(kCholThreads<R>)
cq_chol_kernel(const CqPanel* __restrict__ panels, const float* __restrict__ partial,
               float* __restrict__ linv, uint32_t* __restrict__ status) {
  constexpr int kLd = R + 1, kBlks = R / kNb, kThreads = kCholThreads<R>;
  extern __shared__ float cq_smem[];
  // R x kLd: G, whose lower triangle becomes L below its diagonal blocks; the transpose of L^-1
  // (on the way, of the L L^-1 of rows to come) in the diagonal blocks and above
  float* A = cq_smem;
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
      // Phase 1: the diagonal block, row k0 + lane in lane < 16, and its inverse, a column per lane
      float a[kNb], inv[kNb];
      const int row = lane & (kNb - 1);
#pragma unroll
      for (int j = 0; j < kNb; ++j) a[j] = A[(k0 + row) * kLd + k0 + j];
      bool neg = false;
#pragma unroll
      for (int j = 0; j < kNb; ++j) {
        const float d = __shfl_sync(0xffffffffu, a[j], j);
        neg = neg || !(d > 0.f);
        const float l = sqrtf(d > 0.f ? d : 1.f);
        inv[j] = 1.f / l;
        a[j] = row == j ? l : a[j] * inv[j];
#pragma unroll
        for (int k = 0; k < kNb; ++k) {
          if (k <= j) continue;
          const float lk = __shfl_sync(0xffffffffu, a[j], k);
          if (row >= k) a[k] = fmaf(-a[j], lk, a[k]);
        }
      }
      // L Y = I: lane c solves column c; L's rows come from their lanes
      float y[kNb];
#pragma unroll
      for (int i = 0; i < kNb; ++i) {
        float s = row == i ? 1.f : 0.f;
#pragma unroll
        for (int k = 0; k < kNb; ++k)
          if (k < i) s = fmaf(-__shfl_sync(0xffffffffu, a[k], i), y[k], s);
        y[i] = i >= row ? s * inv[i] : 0.f;
      }
      if (lane < kNb) {
#pragma unroll
        for (int j = 0; j < kNb; ++j) A[(k0 + row) * kLd + k0 + j] = y[j];
      }
      if (neg && lane == 0) bad = 1;
    }
    __syncthreads();
    // Phase 2.  With D = L_11^-1 (its transpose is in A), rows below: L_21 = G_21 D^T (4 of a
    // row's 16 entries an item); columns to the left: L^-1's rows k0 .. are -D times what phase
    // 3 has summed there (4 rows of a column an item).  In place, so computed before written.
    const int n_rows = R - k0 - kNb;
    float v[4] = {0.f, 0.f, 0.f, 0.f};
    float* o = nullptr;
    if (tid < 4 * n_rows) {
      const float* x = A + (k0 + kNb + tid / 4) * kLd + k0;
      const float* y = A + k0 * kLd + k0 + 4 * (tid % 4);
#pragma unroll
      for (int k = 0; k < kNb; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = fmaf(x[k], y[k * kLd + c], v[c]);
      o = A + (k0 + kNb + tid / 4) * kLd + k0 + 4 * (tid % 4);
    } else if (tid < 4 * (n_rows + k0)) {
      const int rq = (tid - 4 * n_rows) / k0, col = (tid - 4 * n_rows) % k0;
      const float* x = A + k0 * kLd + k0 + 4 * rq;
      const float* y = A + col * kLd + k0;
#pragma unroll
      for (int k = 0; k < kNb; ++k)
#pragma unroll
        for (int c = 0; c < 4; ++c) v[c] = fmaf(-x[k * kLd + c], y[k], v[c]);
      o = A + col * kLd + k0 + 4 * rq;
    }
    __syncthreads();
    if (o != nullptr)
#pragma unroll
      for (int c = 0; c < 4; ++c) o[c] = v[c];
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
          for (int j = 0; j < 4; ++j) s[i][j] = 0.f;
#pragma unroll
        for (int k = 0; k < kNb; ++k)
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j <= i) s[i][j] = fmaf(x[i * nt * kLd + k], y[j * nt * kLd + k], s[i][j]);
#pragma unroll
        for (int i = 0; i < 4; ++i)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < i || (j == i && tj <= ti)) g[i * nt * kLd + j * nt] -= s[i][j];
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
// past half of b only the second half's are left.  4 layers of the 32B set at r = 64: 79 us
// (31 for the bytes, 44 for the multiply-adds, 49 for the shared-memory reads).
constexpr int kApplyThreads = 256;
template <int R>
struct Apply {
  static constexpr int kColThreads = R / 8;
  static constexpr int kRowThreads = kApplyThreads / kColThreads;     // 128, 64, 32, 16
  static constexpr int kTR = R == 16 ? 2 : R == 64 ? 8 : 4;           // rows per thread
  static constexpr int kRows = kRowThreads * kTR;                     // 256; 64 at R = 128
  static constexpr int kLd = R + 4;
  static constexpr size_t kSmem = sizeof(float) * ((size_t)kRows + R) * kLd;
};

template <int R>
__global__ void __launch_bounds__(kApplyThreads, R <= 32 ? 3 : 2)
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
  for (int w = tid; w < R * kW; w += kApplyThreads)
    cp_async_16(LT + (w / kW) * kLd + 4 * (w % kW), L + 4 * w, 16);
  for (int s0 = blockIdx.y * Cfg::kRows; s0 < ch.nrows; s0 += gridDim.y * Cfg::kRows) {
    const int n = min(Cfg::kRows, ch.nrows - s0);
    float* rows = pn.out + (ch.row0 + s0) * R;
    __syncthreads();
    for (int w = tid; w < n * kW; w += kApplyThreads)
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
                         uint32_t refresh_idx, uint32_t* d_status, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(cq_chol_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)chol_smem<R>());
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cq_gram_kernel<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Gram<R, true>::kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cq_gram_kernel<R, false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Gram<R, false>::kSmem);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(cq_apply_kernel<R>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)Apply<R>::kSmem);
  if (e != cudaSuccess) return e;
  // CTAs per chunk of 256-row parts: one each, or two parts (L^-1 read half as often)
  const int n_split = R >= 64 || n_chunks < 608 ? cq_chunk_rows(R) / 256 : cq_chunk_rows(R) / 512;
  // first Cholesky QR: Omega -> Q1; second: Q1 -> Q; both in the panels
  for (int round = 0; round < 2; ++round) {
    if (round == 0)
      cq_gram_kernel<R, true><<<n_chunks, Gram<R, true>::kThreads, Gram<R, true>::kSmem, s>>>(
          d_panels, d_chunks, d_partial, seed, refresh_idx);
    else
      cq_gram_kernel<R, false><<<n_chunks, Gram<R, false>::kThreads, Gram<R, false>::kSmem, s>>>(
          d_panels, d_chunks, d_partial, seed, refresh_idx);
    e = launch_dependent(cq_chol_kernel<R>, (unsigned)(n_panels * kCholCtas), kCholThreads<R>,
                         chol_smem<R>(), s, kCholCtas, false, d_panels, d_partial, d_linv, d_status);
    if (e != cudaSuccess) return e;
    cq_apply_kernel<R><<<dim3(n_chunks, n_split), kApplyThreads, Apply<R>::kSmem, s>>>(
        d_panels, d_chunks, d_linv);
  }
  return cudaGetLastError();
}

}  // namespace

bool cholqr_supported(int32_t r) { return r == 16 || r == 32 || r == 64 || r == 128; }

cudaError_t launch_cholqr(const CqPanel* d_panels, int32_t n_panels, const CqChunk* d_chunks,
                          int32_t n_chunks, float* d_partial, float* d_linv, int32_t r,
                          uint64_t seed, uint32_t refresh_idx, uint32_t* d_status, cudaStream_t s) {
  if (n_panels <= 0) return cudaSuccess;
  switch (r) {
    case 16: return run_cholqr_r<16>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, d_status, s);
    case 32: return run_cholqr_r<32>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, d_status, s);
    case 64: return run_cholqr_r<64>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, d_status, s);
    case 128: return run_cholqr_r<128>(d_panels, n_panels, d_chunks, n_chunks, d_partial, d_linv, seed, refresh_idx, d_status, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zo
