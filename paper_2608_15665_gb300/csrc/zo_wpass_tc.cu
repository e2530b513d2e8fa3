// Weight pass on the 5th-generation tensor cores: W_i <- rnd_bf16(W_i + U_i P_i)
// for every bf16 matrix in one persistent launch (the fused form of Alg. 2's
// "W_i <- W_i + eps U_i Z_i V_i^T", Eq. (4), and of the update of Eq. (10)).
// This file holds the kernel for r <= 32 (both operands in shared memory) and the
// dispatch by rank; the r >= 64 kernel, which reads U from Tensor Memory, is in
// zo_wpass_tmem.cu; the U operand is prepared in zo_operands.cu (r <= 32) or
// zo_wpass_tmem.cu (r >= 64), the P operand by zo_project_tc.cu.
//
// The contraction U (128 x r) . P (r x 128) of a 128 x 128 tile is r-deep, so it
// costs 2r flops per weight against 4 bytes of HBM traffic; past r = 16 that is
// more than the fp32 FMA pipes deliver at HBM speed, so it runs on tcgen05.mma.
// To keep fp32-grade accuracy of the update with 16-bit tensor-core inputs, both
// operands are held as power-of-two-scaled fp16 pairs x s = hi + lo (hi = f16(x s),
// lo = f16(x s - hi); the scales in zo_tc_common.cuh) and the tile accumulates
// hi.hi + hi.lo + lo.hi in fp32 in Tensor Memory: relative error of the product
// ~2^-21 of sum |U| |P|, against 2^-16 for a bf16 pair and 2^-8 for plain bf16.  The
// epilogue undoes the scales with one fp32 multiply-add per weight.
//
// Roles of the 224 threads of a CTA (one CTA per SM, persistent over the chunks of 4
// tiles b, b + G, b + 2G, ... of the interleaved walk, G = number of CTAs):
//   warp 0, lane 0: TMA producer of W -- each tile as 8 boxes of 32 rows x 64
//                   columns, 128-byte swizzle, as far ahead as the W ring allows.
//   warp 6, lane 0: TMA producer of the operands -- the U tile when the row block
//                   changes, the P tile of every tile.  Apart from the W producer,
//                   so a W prefetch never queues behind an operand slot that the
//                   MMAs of an earlier tile still hold.
//   warp 1, lane 0: MMA issuer -- 3 * r/16 tcgen05.mma (M=128, N=128, K=16) per
//                   tile into one of two TMEM accumulators; warp 1 also owns
//                   the TMEM allocation.
//   warps 2..5:     epilogue -- each warp owns 32 rows (its TMEM lane group):
//                   tcgen05.ld the fp32 update, scale it and add it to the W rows
//                   in shared memory, round to bf16 in place, TMA-store its rows.
// Every mbarrier wait is bounded; on expiry the kernel records kDevTimeout in
// the status word, lets the other roles stop, drains its copies and frees TMEM.
#include <cuda.h>

#include "zo_kernels.h"
#include "zo_launch.cuh"
#include "zo_sm100.cuh"
#include "zo_tc_common.cuh"

namespace zo {
namespace {

using namespace sm100;
using namespace tc;

constexpr int kThreads = 224;

template <int R>
struct TcCfg {
  static_assert(R == 16 || R == 32, "the shared-memory-operand kernel covers r = 16 and 32");
  static constexpr int kHLW = hl_width(R);
  static constexpr int kPanels = kHLW / 64;
  static constexpr int kOpBytes = kPanels * kPanelBytes;        // one operand tile (hi + lo)
  // 4 W stages of 32 KB, 2 + 2 operand stages of 16 KB: 192 KB
  static constexpr int kWStages = 4;
  static constexpr int kAStages = 2;
  static constexpr int kBStages = 2;
  static constexpr int kKC = R / 16;                            // K chunks of 16
  static constexpr size_t kSmem = (size_t)kWStages * kWStageBytes + (size_t)kAStages * kOpBytes +
                                  (size_t)kBStages * kOpBytes + 1024 /*barriers*/ + 1024 /*align*/;
};

template <int R>
__global__ void __launch_bounds__(kThreads, 1)
wpass_tc_kernel(const __grid_constant__ CUtensorMap tm_a, const __grid_constant__ CUtensorMap tm_b,
                const CUtensorMap* __restrict__ w_maps, const TcMat* __restrict__ mats,
                const float* __restrict__ pinv, int n_mats, int64_t n_tiles,
                uint32_t* __restrict__ status, long long wait_cycles, int inject_wait) {
  using Cfg = TcCfg<R>;
  static_assert(Cfg::kWStages >= 2 && Cfg::kWStages <= 4, "W ring must fit Shared::w_full");
  static_assert(Cfg::kAStages >= 1 && Cfg::kAStages <= 2, "A ring must fit Shared::a_full");
  static_assert(Cfg::kBStages >= 1 && Cfg::kBStages <= 2, "B ring must fit Shared::b_full");
  static_assert(sizeof(Shared) <= 1024, "barrier block");
  static_assert(Cfg::kSmem <= 227 * 1024, "shared memory per CTA");
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  uint8_t* w_smem = smem;
  uint8_t* a_smem = w_smem + Cfg::kWStages * kWStageBytes;
  uint8_t* b_smem = a_smem + Cfg::kAStages * Cfg::kOpBytes;
  Shared& sh = *reinterpret_cast<Shared*>(b_smem + Cfg::kBStages * Cfg::kOpBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // Interleaved walk: CTA b takes the chunks of kTileChunk tiles b, b + G, b + 2G, ...
  // At any moment the G CTAs work on neighbouring tiles -- the same row blocks of one
  // matrix -- so the DRAM sees one moving front of nearby rows instead of G scattered
  // streams (LLaMA-7B set: 6.35 TB/s against 5.03 TB/s for contiguous per-CTA ranges);
  // the U tile is reused within a chunk and otherwise reloaded from L2.
  const int64_t G = gridDim.x;
  const int64_t t_begin = (int64_t)blockIdx.x * kTileChunk;
  const int64_t t_end = n_tiles;
  const int64_t t_stride = G * kTileChunk;
  const volatile int* abort = &sh.abort_flag;

  if (threadIdx.x == 0) {
    for (int s = 0; s < Cfg::kWStages; ++s) {
      mbar_init(&sh.w_full[s], 1);
      mbar_init(&sh.w_empty[s], 4);
    }
    for (int s = 0; s < Cfg::kAStages; ++s) {
      mbar_init(&sh.a_full[s], 1);
      mbar_init(&sh.a_empty[s], 1);
    }
    for (int s = 0; s < Cfg::kBStages; ++s) {
      mbar_init(&sh.b_full[s], 1);
      mbar_init(&sh.b_empty[s], 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(&sh.acc_full[s], 1);
      mbar_init(&sh.acc_empty[s], 4);
    }
    mbar_init(&sh.never, 1);
    sh.abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(&tm_a);
    prefetch_tmap(&tm_b);
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_base, 2 * kBN);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  pdl_wait();                              // (no early trigger: see zo_launch.cuh)

  if (warp == 0 && lane == 0) {
    // ------------------------------------------------------------ TMA producer: W tiles
    int64_t n_w = 0;                              // copies issued into the W ring
    bool ok = true;
    TileIter ti;
    ti.init(mats, n_mats, t_begin, t_end, t_stride);
    ti.chunk = kTileChunk;
    for (; ti.valid(); ti.next()) {
      const CUtensorMap* wmap = w_maps + ti.i;
      // W tile: 4 row groups x 2 column halves
      {
        const int s = (int)(n_w % Cfg::kWStages);
        const uint32_t ph = (uint32_t)((n_w / Cfg::kWStages) & 1);
        if (!mbar_wait_bounded(&sh.w_empty[s], ph ^ 1u, abort, wait_cycles)) { ok = false; break; }
        // the tile's scale rides with its W stage: the epilogue warps, which set the pace,
        // then read it from shared memory instead of waiting on a global load
        sh.w_scale[s] = pinv[ti.i] * exp2i(-kUVScaleExp);
        mbar_arrive_expect_tx(&sh.w_full[s], kWStageBytes);
        uint8_t* dst = w_smem + s * kWStageBytes;
        for (int g = 0; g < 4; ++g)
          for (int h = 0; h < 2; ++h)
            tma_load_2d(dst + (g * 2 + h) * kWBoxBytes, wmap, (int)(ti.cb * kBN + 64 * h),
                        (int)(ti.rb * kBM + 32 * g), &sh.w_full[s]);
        ++n_w;
      }
    }
    if (!ok) give_up(sh, status);
    // drain: the last copy issued into every slot has landed before the CTA exits
    for (int s = 0; s < Cfg::kWStages; ++s) {
      const int64_t k = last_in_slot(n_w, s, Cfg::kWStages);
      if (k >= 0) mbar_wait_bounded(&sh.w_full[s], (uint32_t)((k / Cfg::kWStages) & 1), nullptr, wait_cycles);
    }
  } else if (warp == 6 && lane == 0) {
    // ------------------------------------------------------------ TMA producer: operands
    int64_t n_a = 0, n_b = 0;                     // operand tiles issued into each ring
    int64_t a_iss[2] = {0, 0}, b_iss[2] = {0, 0};  // phases issued per barrier
    int prev_i = -1;
    int64_t prev_rb = -1;
    bool ok = true;
    TileIter ti;
    ti.init(mats, n_mats, t_begin, t_end, t_stride);
    ti.chunk = kTileChunk;
    for (; ti.valid(); ti.next()) {
      const TcMat& mt = mats[ti.i];
      // U operand tile once per row block, P operand tile of this column block
      if (ti.i != prev_i || ti.rb != prev_rb) {
        const int sa = (int)(n_a % Cfg::kAStages);
        const uint32_t pa = (uint32_t)((n_a / Cfg::kAStages) & 1);
        if (!mbar_wait_bounded(&sh.a_empty[sa], pa ^ 1u, abort, wait_cycles)) { ok = false; break; }
        mbar_arrive_expect_tx(&sh.a_full[sa], Cfg::kOpBytes);
        ++a_iss[sa];
        for (int p = 0; p < Cfg::kPanels; ++p)
          tma_load_2d(a_smem + sa * Cfg::kOpBytes + p * kPanelBytes, &tm_a, 64 * p,
                      (int)(mt.u_row0 + ti.rb * kBM), &sh.a_full[sa]);
        ++n_a;
        prev_i = ti.i;
        prev_rb = ti.rb;
      }
      const int sb = (int)(n_b % Cfg::kBStages);
      const uint32_t pb = (uint32_t)((n_b / Cfg::kBStages) & 1);
      if (!mbar_wait_bounded(&sh.b_empty[sb], pb ^ 1u, abort, wait_cycles)) { ok = false; break; }
      mbar_arrive_expect_tx(&sh.b_full[sb], Cfg::kOpBytes);
      ++b_iss[sb];
      for (int p = 0; p < Cfg::kPanels; ++p)
        tma_load_2d(b_smem + sb * Cfg::kOpBytes + p * kPanelBytes, &tm_b, 64 * p,
                    (int)(mt.p_row0 + ti.cb * kBN), &sh.b_full[sb]);
      ++n_b;
    }
    if (!ok) give_up(sh, status);
    // drain: the last phase issued on every operand barrier has landed before the CTA exits
    for (int bi = 0; bi < Cfg::kAStages; ++bi)
      if (a_iss[bi] > 0)
        mbar_wait_bounded(&sh.a_full[bi], (uint32_t)((a_iss[bi] - 1) & 1), nullptr, wait_cycles);
    for (int bi = 0; bi < Cfg::kBStages; ++bi)
      if (b_iss[bi] > 0)
        mbar_wait_bounded(&sh.b_full[bi], (uint32_t)((b_iss[bi] - 1) & 1), nullptr, wait_cycles);
  } else if (warp == 1 && lane == 0) {
    // ------------------------------------------------------------ MMA issuer
    constexpr uint32_t idesc = idesc_f16_f32(kBM, kBN);
    int64_t it = 0, a_it = 0;
    int prev_i = -1;
    int64_t prev_rb = -1;
    int sa = 0;
    bool ok = true;
    TileIter ti, nx;                            // nx runs one tile ahead of ti
    ti.init(mats, n_mats, t_begin, t_end, t_stride);
    ti.chunk = kTileChunk;
    nx = ti;
    nx.next();
    for (; ti.valid(); ti = nx, nx.next(), ++it) {
      const bool new_a = ti.i != prev_i || ti.rb != prev_rb;
      uint32_t pa = 0;
      if (new_a) {
        sa = (int)(a_it % Cfg::kAStages);
        pa = (uint32_t)((a_it / Cfg::kAStages) & 1);
        ++a_it;
        prev_i = ti.i;
        prev_rb = ti.rb;
      }
      // the U tile is released after its last tile: the next tile starts another row
      // block (or there is none)
      const bool last_a = !nx.valid() || nx.i != ti.i || nx.rb != ti.rb;
      const int sb = (int)(it % Cfg::kBStages);
      const uint32_t pb = (uint32_t)((it / Cfg::kBStages) & 1);
      const int acc = (int)(it & 1);
      if (!mbar_wait_bounded(&sh.acc_empty[acc], (uint32_t)(((it >> 1) & 1) ^ 1), abort,
                             wait_cycles)) { ok = false; break; }
      const uint32_t d = tmem + (uint32_t)(acc * kBN);
      const uint32_t a_base = smem_u32(a_smem + sa * Cfg::kOpBytes);
      const uint32_t b_base = smem_u32(b_smem + sb * Cfg::kOpBytes);
      if (new_a && !mbar_wait_bounded(&sh.a_full[sa], pa, abort, wait_cycles)) {
        ok = false;
        break;
      }
      if (!mbar_wait_bounded(&sh.b_full[sb], pb, abort, wait_cycles)) {
        ok = false;
        break;
      }
      tc_fence_after();
      // the small cross products hi.lo and lo.hi first, hi.hi last: each MMA adds its
      // products to the fp32 accumulator with one rounding relative to the accumulator's
      // magnitude, so only the r/16 hi.hi MMAs round at the update's full size
#pragma unroll
      for (int pass = 0; pass < 3; ++pass) {
#pragma unroll
        for (int kk = 0; kk < Cfg::kKC; ++kk) {
          // hi chunk kk at element 16 kk of the operand row, lo chunk at R + 16 kk
          const int e_hi = 16 * kk, e_lo = R + 16 * kk;
          const uint32_t off_hi = (uint32_t)((e_hi / 64) * kPanelBytes + (e_hi % 64) * 2);
          const uint32_t off_lo = (uint32_t)((e_lo / 64) * kPanelBytes + (e_lo % 64) * 2);
          const uint64_t a_d = sdesc_k_sw128(a_base + (pass == 1 ? off_lo : off_hi));
          const uint64_t b_d = sdesc_k_sw128(b_base + (pass == 0 ? off_lo : off_hi));
          mma_f16(d, a_d, b_d, idesc, (pass | kk) != 0 ? 1u : 0u);
        }
      }
      mma_commit(&sh.b_empty[sb]);
      if (last_a) mma_commit(&sh.a_empty[sa]);
      mma_commit(&sh.acc_full[acc]);
    }
    if (!ok) give_up(sh, status);
    if (it > 0) {
      // every MMA issued by this thread has completed before TMEM is released
      const int64_t last = it - 1;
      mbar_wait_bounded(&sh.acc_full[last & 1], (uint32_t)((last >> 1) & 1), nullptr, wait_cycles);
    }
  } else if (warp >= 2 && warp <= 5) {
    // ------------------------------------------------------------ epilogue
    const int g = warp & 3;                      // TMEM lane group == tile row group
    const uint32_t lane_base = (uint32_t)(g * 32) << 16;
    int64_t it = 0;
    bool ok = true;
    TileIter ti;
    ti.init(mats, n_mats, t_begin, t_end, t_stride);
    ti.chunk = kTileChunk;
    for (; ti.valid(); ti.next(), ++it) {
      const TcMat& mt = mats[ti.i];
      const int acc = (int)(it & 1);
      // test hook (zo_set_option ZO_OPTION_TEST_WAIT_TIMEOUT): CTA 0's epilogue first waits
      // on a barrier that nothing arrives on, so its bounded wait runs out
      if (inject_wait && blockIdx.x == 0 && it == 0 &&
          !mbar_wait_bounded(&sh.never, 0u, abort, wait_cycles)) {
        ok = false;
        break;
      }
      if (!mbar_wait_bounded(&sh.acc_full[acc], (uint32_t)((it >> 1) & 1), abort, wait_cycles)) {
        ok = false;
        break;
      }
      tc_fence_after();
      const int s = (int)(it % Cfg::kWStages);
      if (!mbar_wait_bounded(&sh.w_full[s], (uint32_t)((it / Cfg::kWStages) & 1), abort,
                             wait_cycles)) {
        ok = false;
        break;
      }
      uint8_t* stage = w_smem + s * kWStageBytes;
      // the accumulator holds 2^(kUVScaleExp + e_P,i) U P: back to U P in the add
      const uint64_t wscale2 = splat2(sh.w_scale[s]);
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        uint32_t v[32];
        tmem_ld_32x32b_x32(tmem + lane_base + (uint32_t)(acc * kBN + c * 32), v);
        tmem_ld_wait();
        uint8_t* box = stage + (g * 2 + (c >> 1)) * kWBoxBytes + lane * 128;
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          const int j = (c & 1) * 4 + j4;                       // logical 16-byte chunk
          uint4* p = reinterpret_cast<uint4*>(box + ((j ^ (lane & 7)) << 4));
          uint4 raw = *p;
          uint32_t wv[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
          for (int e = 0; e < 4; ++e)
            wv[e] = bf16x2_add_scaled(wv[e], v[j4 * 8 + 2 * e], v[j4 * 8 + 2 * e + 1], wscale2);
          *p = make_uint4(wv[0], wv[1], wv[2], wv[3]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&sh.acc_empty[acc]);
      fence_async_smem();
      __syncwarp();
      if (lane == 0) {
        const int64_t y = ti.rb * kBM + 32 * g;
        if (y < mt.m) {
          for (int h = 0; h < 2; ++h) {
            const int64_t x = ti.cb * kBN + 64 * h;
            if (x < mt.n)
              tma_store_2d(w_maps + ti.i, (int)x, (int)y, stage + (g * 2 + h) * kWBoxBytes);
          }
        }
        bulk_commit();
        bulk_wait_read_all();
        mbar_arrive(&sh.w_empty[s]);
      }
      __syncwarp();
    }
    if (!ok && lane == 0) give_up(sh, status);
    if (lane == 0) bulk_wait_all();
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 2 * kBN);
  }
}

template <int R>
cudaError_t launch_tc_r(const CUtensorMap& tm_a, const CUtensorMap& tm_b, const CUtensorMap* w_maps,
                        const TcMat* mats, const float* pinv, int n_mats, int64_t n_tiles, int grid,
                        uint32_t* status, bool inject_wait, cudaStream_t s) {
  const size_t smem = TcCfg<R>::kSmem;
  cudaError_t e = cudaFuncSetAttribute(wpass_tc_kernel<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  // with the test hook armed the wait limit is ~0.1 s so the test ends quickly
  const long long wait = inject_wait ? kTestWaitCycles : kWaitCycles;
  return launch_dependent(wpass_tc_kernel<R>, (unsigned)grid, kThreads, smem, s, 1, true, tm_a, tm_b,
                          w_maps, mats, pinv, n_mats, n_tiles, status, wait, inject_wait ? 1 : 0);
}

}  // namespace

bool wpass_tc_supported(int32_t r) { return r == 16 || r == 32 || r == 64 || r == 128; }
bool wpass_tc_u_in_tmem(int32_t r) { return r >= 64; }
int32_t tc_hl_width(int32_t r) { return hl_width(r); }
int32_t tc_tile_rows() { return kBM; }
int32_t tc_tile_cols() { return kBN; }
int64_t tc_u_operand_bytes(int32_t r, int64_t rows) {
  const int64_t row_layout = rows * hl_width(r) * 2;        // 16-bit [hi | lo | 0] rows
  const int64_t chunk_layout = rows * r * 4;                // R 32-bit words per row
  return row_layout > chunk_layout ? row_layout : chunk_layout;
}

cudaError_t launch_wpass_tc(const CUtensorMap& tm_a, const void* u_op, const CUtensorMap& tm_b,
                            const CUtensorMap* d_w_maps, const TcMat* d_tc, const float* d_pinv,
                            int32_t n_mats, int64_t n_tiles, int32_t grid, int32_t r,
                            uint32_t* d_status, bool inject_wait, cudaStream_t s) {
  if (n_tiles <= 0) return cudaSuccess;
  switch (r) {
    case 16: return launch_tc_r<16>(tm_a, tm_b, d_w_maps, d_tc, d_pinv, n_mats, n_tiles, grid, d_status, inject_wait, s);
    case 32: return launch_tc_r<32>(tm_a, tm_b, d_w_maps, d_tc, d_pinv, n_mats, n_tiles, grid, d_status, inject_wait, s);
    case 64:
    case 128:
      return launch_wpass_tmem(static_cast<const uint4*>(u_op), tm_b, d_w_maps, d_tc, d_pinv, n_mats,
                               n_tiles, grid, r, d_status, inject_wait, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace zo
