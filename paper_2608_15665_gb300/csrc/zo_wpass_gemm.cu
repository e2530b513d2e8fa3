// Weight pass, fp32-FMA path, on 64 x 128 tiles: W_i <- rnd(W_i + U_i P_i) with
// P_i = C_i V_i^T precomputed (r x n fp32), for fp32 weights, bf16 weights whose width is
// not a multiple of 8, and r <= 8 sets too large for the one-launch kernels of
// zo_wpass_fma.cu.  Each term is one fp32 multiply-add from zero in ascending k, then one
// add and one rounding into W: the arithmetic of those kernels, so all FMA tilings give the
// same bits.
//
// Bound: reading and writing W up to r = 32 (85 M fp32 weights: 100 us of HBM, 70 us of FMA
// at r = 32), FMA issue above.  What the layout is for:
//  * 16 x 16 threads of a 4 x 8 register tile.  The 4 x 4 tile of a 32-row kernel with P
//    staged through registers took 493 us for those weights at r = 32 and 2604 us at
//    r = 128; this kernel takes 164 and 482 us (bf16: 397 -> 148 us at r = 32).
//  * Two multiply-adds per instruction (fma.rn.f32x2): plain fmaf measured 196 us at r = 32
//    and 558 us at r = 128 on 128-row tiles, packed 176 and 473 us.
//  * Everything is copied by cp.async: the U rows and P columns in chunks of 16 k, two chunks
//    in flight, and the tile's W behind them, so that W's HBM latency passes under the FMAs.
//    Three CTAs per SM overlap one's loads and stores with the others' arithmetic: at
//    r = 32 and 64 that makes 64-row tiles faster than 128-row ones with two CTAs (164 and
//    267 us against 176 and 295), elsewhere they are within 3%; 32-row tiles are slower
//    (217 and 385 us).  At r <= 16, where there is little arithmetic to hide W's latency under,
//    four CTAs, at 64 registers, although r = 16 then spills (32 bytes stored, 76 loaded; r = 4 12
//    and 32, r = 8 nothing): 121 -> 115 us at r = 16, 112 -> 105 at r = 8 (bf16: 85 -> 77).  Five
//    or six spill far more (160 and 245 us at r = 8).  From r = 32 on, fewer, 8 x 8 register tiles
//    read less from shared memory, of which the 4 x 8 ones take 67%, but leave too few warps
//    (128 threads: 192 us at r = 32).
#include "zo_fma_common.cuh"
#include "zo_launch.cuh"

namespace zo {
namespace {

using namespace fma;

constexpr int kGemmThreads = 256;
constexpr int kGemmRows = kGemmTileRows;   // 64
constexpr int kGemmCols = kGemmTileCols;   // 128

template <int R>
struct GemmShape {
  static constexpr int kC = R < 16 ? R : 16;          // k per chunk
  static constexpr int kChunks = R / kC;
  static constexpr int kStages = kChunks < 2 ? kChunks : 2;
  // a U row's pitch: the two rows a warp reads at once fall into different banks
  static constexpr int kLdU = kC + 4;
  static constexpr int kStageFloats = kGemmRows * kLdU + kC * kGemmCols;
  static constexpr size_t kSmem =
      sizeof(float) * ((size_t)kStages * kStageFloats + (size_t)kGemmRows * kGemmCols);
};

__device__ __forceinline__ void add_store(float* w, const float* ws, const float (&acc)[4]) {
  float4 x = *reinterpret_cast<const float4*>(ws);
  x.x += acc[0]; x.y += acc[1]; x.z += acc[2]; x.w += acc[3];
  *reinterpret_cast<float4*>(w) = x;
}
__device__ __forceinline__ void add_store(__nv_bfloat16* w, const __nv_bfloat16* ws,
                                          const float (&acc)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(ws);
  uint2 o;
  o.x = pack2_bf16(__uint_as_float(v.x << 16) + acc[0], __uint_as_float(v.x & 0xFFFF0000u) + acc[1]);
  o.y = pack2_bf16(__uint_as_float(v.y << 16) + acc[2], __uint_as_float(v.y & 0xFFFF0000u) + acc[3]);
  *reinterpret_cast<uint2*>(w) = o;
}

template <int R, typename T>
__device__ __forceinline__ void gemm_tile(const MatDesc& md, int64_t local, float* smem) {
  using S = GemmShape<R>;
  constexpr int KC = S::kC, LDU = S::kLdU, VEC = Vec<T>::N;
  constexpr int BM = kGemmRows, TR = BM / 16;         // TR rows per thread
  constexpr int kStage = S::kStageFloats;
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int64_t m = md.m, n = md.n;
  const int64_t tiles_n = (n + kGemmCols - 1) / kGemmCols;
  const int64_t row0 = (local / tiles_n) * BM, col0 = (local % tiles_n) * kGemmCols;
  T* W = reinterpret_cast<T*>(md.W);
  T* Ws = reinterpret_cast<T*>(smem + S::kStages * kStage);
  const bool p_vec = (n & 3) == 0;                    // P's rows are n floats apart

  auto load_chunk = [&](int c) {
    float* Us = smem + (c % S::kStages) * kStage;
    float* Ps = Us + BM * LDU;
#pragma unroll
    for (int idx = tid; idx < BM * KC / 4; idx += kGemmThreads) {
      const int row = idx / (KC / 4), k4 = idx % (KC / 4);
      const bool live = row0 + row < m;
      cp_async_16(Us + row * LDU + 4 * k4,
                  md.U + (live ? (row0 + row) * R + c * KC + 4 * k4 : 0), live ? 16 : 0);
    }
    if (p_vec) {
#pragma unroll
      for (int idx = tid; idx < KC * kGemmCols / 4; idx += kGemmThreads) {
        const int k = idx / (kGemmCols / 4), c4 = idx % (kGemmCols / 4);
        const int64_t col = col0 + 4 * c4;
        const bool live = col < n;
        cp_async_16(Ps + k * kGemmCols + 4 * c4, md.P + (live ? (c * KC + k) * n + col : 0),
                    live ? 16 : 0);
      }
    } else {
#pragma unroll
      for (int idx = tid; idx < KC * kGemmCols; idx += kGemmThreads) {
        const int k = idx / kGemmCols, cc = idx % kGemmCols;
        const bool live = col0 + cc < n;
        cp_async_4(Ps + k * kGemmCols + cc, md.P + (live ? (c * KC + k) * n + col0 + cc : 0),
                   live ? 4 : 0);
      }
    }
  };

  load_chunk(0);
  cp_async_commit();
  if (S::kChunks > 1) load_chunk(1);
  cp_async_commit();
  // the tile's W; the last, partial 16 bytes of a row are read only up to its n elements
  constexpr int kRowVecs = kGemmCols / VEC;
#pragma unroll
  for (int idx = tid; idx < BM * kRowVecs; idx += kGemmThreads) {
    const int row = idx / kRowVecs, v = idx % kRowVecs;
    const int64_t col = col0 + v * VEC;
    const int64_t left = row0 + row < m ? n - col : 0;
    const int bytes = left >= VEC ? 16 : left > 0 ? (int)left * (int)sizeof(T) : 0;
    cp_async_16(Ws + row * kGemmCols + v * VEC, W + (bytes ? (row0 + row) * md.ldw + col : 0),
                bytes);
  }
  cp_async_commit();

  float2 acc[TR][4];                                  // column pairs
#pragma unroll
  for (int i = 0; i < TR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = make_float2(0.f, 0.f);

#pragma unroll
  for (int c = 0; c < S::kChunks; ++c) {
    // copies committed after chunk c's: chunk 1 and W (c = 0), W and chunk 2 (c = 1), else
    // chunk c + 1
    if (c < 2) cp_async_wait<2>();
    else cp_async_wait<1>();
    __syncthreads();
    const float* Us = smem + (c % S::kStages) * kStage + ty * LDU;
    const float* Ps = smem + (c % S::kStages) * kStage + BM * LDU + 4 * tx;
#pragma unroll
    for (int k2 = 0; k2 < KC / 2; ++k2) {
      float2 u[TR];
#pragma unroll
      for (int i = 0; i < TR; ++i)
        u[i] = *reinterpret_cast<const float2*>(Us + 16 * i * LDU + 2 * k2);
#pragma unroll
      for (int kk = 0; kk < 2; ++kk) {
        const float4 a = *reinterpret_cast<const float4*>(Ps + (2 * k2 + kk) * kGemmCols);
        const float4 b = *reinterpret_cast<const float4*>(Ps + (2 * k2 + kk) * kGemmCols + 64);
        const float2 p[4] = {make_float2(a.x, a.y), make_float2(a.z, a.w), make_float2(b.x, b.y),
                             make_float2(b.z, b.w)};
#pragma unroll
        for (int i = 0; i < TR; ++i) {
          const float uk = kk == 0 ? u[i].x : u[i].y;
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[i][j] = fma2(make_float2(uk, uk), p[j], acc[i][j]);
        }
      }
    }
    if (c + 2 < S::kChunks) {
      __syncthreads();                                // every warp is done with this stage
      load_chunk(c + 2);
    }
    cp_async_commit();                                // possibly empty: keeps the count
  }
  cp_async_wait<0>();
  __syncthreads();

#pragma unroll
  for (int i = 0; i < TR; ++i) {
    const int64_t row = row0 + ty + 16 * i;
    if (row >= m) continue;
    T* wrow = W + row * md.ldw;
#pragma unroll
    for (int g = 0; g < 2; ++g) {
      const int64_t col = col0 + 64 * g + 4 * tx;
      const T* ws = Ws + (ty + 16 * i) * kGemmCols + 64 * g + 4 * tx;
      const float d[4] = {acc[i][2 * g].x, acc[i][2 * g].y, acc[i][2 * g + 1].x,
                          acc[i][2 * g + 1].y};
      if (col + 4 <= n) {
        add_store(wrow + col, ws, d);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (col + e < n) store_scalar<T>(wrow + col + e, load_scalar<T>(ws + e) + d[e]);
      }
    }
  }
}

template <int R>
__global__ void __launch_bounds__(kGemmThreads, R <= 16 ? 4 : 3)
wpass_gemm_kernel(const MatDesc* __restrict__ mats, int n_mats, const int64_t* __restrict__ prefix) {
  extern __shared__ float4 smem4[];
  float* smem = reinterpret_cast<float*>(smem4);
  const int64_t tile = blockIdx.x;
  const int i = find_matrix(prefix, n_mats, tile);
  const MatDesc md = mats[i];
  const int64_t local = tile - __ldg(prefix + i);
  pdl_wait();
  pdl_trigger();
  if (md.dtype == 1)
    gemm_tile<R, __nv_bfloat16>(md, local, smem);
  else
    gemm_tile<R, float>(md, local, smem);
}

template <int R>
cudaError_t launch_gemm_r(const MatDesc* d_mats, int32_t n_mats, const int64_t* d_prefix,
                          int64_t n_tiles, cudaStream_t s) {
  constexpr size_t smem = GemmShape<R>::kSmem;
  cudaError_t e = cudaFuncSetAttribute(wpass_gemm_kernel<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(wpass_gemm_kernel<R>, (unsigned)n_tiles, kGemmThreads, smem, s, 1, true,
                          d_mats, n_mats, d_prefix);
}

}  // namespace

int64_t wpass_gemm_tiles(int64_t m, int64_t n) {
  return (m + kGemmRows - 1) / kGemmRows * ((n + kGemmCols - 1) / kGemmCols);
}

cudaError_t launch_wpass_gemm(const MatDesc* d_mats, int32_t n_mats, const int64_t* d_prefix,
                              int64_t n_tiles, int32_t r, cudaStream_t s) {
  if (n_tiles <= 0) return cudaSuccess;
  if (n_tiles > 0x7FFFFFFF) return cudaErrorInvalidValue;
  switch (r) {
    case 4: return launch_gemm_r<4>(d_mats, n_mats, d_prefix, n_tiles, s);
    case 8: return launch_gemm_r<8>(d_mats, n_mats, d_prefix, n_tiles, s);
    case 16: return launch_gemm_r<16>(d_mats, n_mats, d_prefix, n_tiles, s);
    case 32: return launch_gemm_r<32>(d_mats, n_mats, d_prefix, n_tiles, s);
    case 64: return launch_gemm_r<64>(d_mats, n_mats, d_prefix, n_tiles, s);
    case 128: return launch_gemm_r<128>(d_mats, n_mats, d_prefix, n_tiles, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zo
