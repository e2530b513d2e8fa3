// The perturbed linear layer (Y = X W_i^T + S U_i^T, S = X P^T, the forward of Alg. 3 at
// W' = W + eps U Z V^T, Eq. (4) form, with W left as it is) for at most 128 tokens at r <= 64, where
// reading W_i is what there is to do.
//
// One CTA per SM owns all the tokens and `cols` columns of Y (rows of W_i; a multiple of 16
// chosen so that m / cols CTAs fill the SMs once): an M = 128 tcgen05.mma with the tokens as
// its rows and the W rows as its N columns, over all of K.  The SM-pair tiles of
// zo_linear_pair.cu compute 256 x 128 or more whatever the tokens, on m / 128 of the 76 pairs
// at most, and so stream W through a part of the SMs.  Only the tokens' rows of X are loaded;
// the MMA's rows past them read whatever follows in shared memory and end in accumulator
// lanes that nothing reads.
//
// S = X P^T comes from the first CTAs of the grid, one per 32 tokens and 32 (16 at r = 16)
// columns of S, each over all of K with a smaller operand stream than the others', so that S
// is there when they are done with W: they write S_HL's rows and set a ready flag, and the
// others' producers wait for all flags before the rank-r step.  They are dispatched first and
// wait on nothing, so the waits cannot block the grid.
//
// K steps and the rank-r step's products are those of the SM-pair kernel, in its order, with
// one accumulator per output: Y has its bits.  (At r = 128 that kernel sums S over ranges of K
// in fp32; one range here moved Y by up to rel 3.3e-5, so r = 128 stays with it, although
// 4096 x 4096 took 18, 20 and 20 us at 1, 97 and 128 tokens here and takes 36, 53 and 60.)
//
// Bound: an output's chain of MMAs, about 85 cycles for each 16 elements of K however few the
// columns (1024 x 12288: 38 us at any T), until the stream into the SM, 128 B per token and W
// row for 64 elements of K, or HBM's 2 bytes per weight take longer (12288 x 12288: 49 us at
// one token, 6.2 TB/s).  Measured at 1, 97 and 128 tokens, r = 32, against the SM-pair kernel's
// best tiling: 4096 x 4096 17.6, 17.3, 17.3 us (28, 26, 26); 11008 x 4096 19.4, 20.2, 22.5 us
// (41, 28, 29); 4096 x 11008 35, 37, 37 us (55, 54, 54).  Over 13 shapes from 264 x 136 to 12288 x
// 768 and 768 x 12288, r = 16, 32 and 64 and 1 to 128 tokens it takes 0.41 to 0.80 of that kernel's
// time, least ahead on tall W at 128 tokens.  Short K at 1, 32, 128 tokens: 512 x 512 at r = 16 6.6,
// 6.7, 7.1 us (10.4, 10.6, 11.3), at r = 64 6.9, 7.0, 7.5 (11.0, 11.3, 11.7); 4096 x 512 at r = 16
// 7.2, 7.4, 8.0 (10.9, 11.2, 11.5), at r = 64 7.9, 8.1, 8.8 (12.6, 12.5, 13.2); 16384 x 512 at r = 32
// 8.9, 9.4, 9.8 (12.0, 12.1, 12.6).  Splitting K over a cluster of CTAs
// cuts the chain (4096 x 11008: 19 us at one token) but sums in another order, and its exchange
// grows with the tokens (25 us at 97).
//
// Roles (256 threads): warp 0 lane 0 loads by TMA, warp 1 lane 0 issues the MMAs (warp 1 owns
// the Tensor Memory), then all eight warps empty the accumulator.  Every wait is bounded; a
// give-up sets kDevTimeout, the producer waits for its copies in flight, the MMA thread for
// its MMAs, and TMEM is freed.
#include <algorithm>

#include <cuda.h>

#include "zo_kernels.h"
#include "zo_launch.cuh"
#include "zo_linear_common.cuh"
#include "zo_sm100.cuh"
#include "zo_tc_common.cuh"

namespace zo {
namespace {

using namespace sm100;
using namespace tc;
using namespace lin;

constexpr int kMaxTokens = 128;
constexpr int kSTokens = 32;             // tokens of one CTA of S
constexpr int kThreads = 256;
constexpr int kMaxStages = 12;
constexpr int kTmemCols = 128;
constexpr int kASpan = 128 * 128;        // bytes of A that an MMA reads, whatever is loaded

__host__ __device__ constexpr int s_cols(int r) { return r < 32 ? r : 32; }   // of one CTA of S

struct FewShared {
  uint64_t full[kMaxStages], empty[kMaxStages];
  uint64_t acc_full;
  uint32_t tmem_base;
  int abort_flag;
};

struct FewArgs {
  int T, m;                // tokens, columns of Y
  int tokens;              // T rounded up to 16: rows of the X and S_HL boxes
  int cols;                // columns of Y per CTA (MMA N), a multiple of 16
  int k_steps;             // 64-element panels of K
  int n_s;                 // CTAs of S
  int panels, s_panels;    // 64-element panels of K per operand stage of the Y and the S CTAs
  int stages, s_stages;
  int u_row0;
  int64_t ldy;
  __nv_bfloat16* Y;
  __nv_bfloat16* s_hl;
  uint32_t* flags;         // one per CTA of S
  uint32_t epoch, wait_epoch;
  uint32_t* status;
  long long wait_cycles;
};

// tm_x: X (box 64 x tokens), tm_xs: X (box 64 x kSTokens), tm_w: W_i (box 64 x cols), tm_pk:
// P_K (box 64 x s_cols(R)), tm_s: S_HL (box 64 x tokens), tm_u: the route's U operand
// (box 64 x cols; this matrix's rows from u_row0).
template <int R>
__global__ void __launch_bounds__(kThreads, 1)
linear_few_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_xs,
                  const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_pk,
                  const __grid_constant__ CUtensorMap tm_s, const __grid_constant__ CUtensorMap tm_u,
                  const FewArgs a) {
  constexpr int kSC = s_cols(R);
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  __shared__ FewShared sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool is_s = (int)blockIdx.x < a.n_s;
  // a panel: its rows of X (or S_HL), then of W (or U, or P_hi and P_lo)
  const int a_rows = is_s ? kSTokens : a.tokens, b_rows = is_s ? 2 * kSC : a.cols;
  const int a_panel = a_rows * 128, b_panel = b_rows * 128;
  const int panels = is_s ? a.s_panels : a.panels;
  const int sbytes = panels * (a_panel + b_panel);
  const int S = is_s ? a.s_stages : a.stages;
  const int s_tok = is_s ? (int)blockIdx.x / (R / kSC) * kSTokens : 0;   // S: first token
  const int s_blk = is_s ? (int)blockIdx.x % (R / kSC) : 0;              // S: block of columns
  const int col0 = is_s ? 0 : ((int)blockIdx.x - a.n_s) * a.cols;
  const int k_stages = (a.k_steps + panels - 1) / panels;
  const int n_k = is_s ? k_stages : k_stages + 1;         // and the rank-r step

  if (threadIdx.x == 0) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    mbar_init(&sh.acc_full, 1);
    sh.abort_flag = 0;
    fence_mbar_init();
    prefetch_tmap(is_s ? &tm_xs : &tm_x);
    prefetch_tmap(is_s ? &tm_pk : &tm_w);
    if (!is_s) {
      prefetch_tmap(&tm_s);
      prefetch_tmap(&tm_u);
    }
  }
  if (warp == 1) {
    tmem_alloc(&sh.tmem_base, kTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  // a programmatic dependent of the stream's previous kernel: everything below may touch
  // memory that kernel writes
  pdl_wait();
  pdl_trigger();
  const volatile int* abort = &sh.abort_flag;

  if (warp == 0 && lane == 0) {
    // ---------------------------------------------------------------- TMA producer
    int s = 0;
    int64_t n_st = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int k = 0; k < n_k && ok; ++k) {
      if (!mbar_wait_bounded(&sh.empty[s], ph ^ 1u, abort, a.wait_cycles)) {
        ok = false;
        break;
      }
      uint8_t* ap = smem + s * sbytes;
      uint8_t* bp = ap + panels * a_panel;
      if (k < k_stages) {
        const int np = min(panels, a.k_steps - panels * k);
        mbar_arrive_expect_tx(&sh.full[s], (uint32_t)(np * (a_panel + b_panel)));
        for (int p = 0; p < np; ++p) {
          const int x = 64 * (panels * k + p);
          if (is_s) {
            tma_load_2d(ap + p * a_panel, &tm_xs, x, s_tok, &sh.full[s]);
            tma_load_2d(bp + p * b_panel, &tm_pk, x, s_blk * kSC, &sh.full[s]);
            tma_load_2d(bp + p * b_panel + kSC * 128, &tm_pk, x, R + s_blk * kSC, &sh.full[s]);
          } else {
            tma_load_2d(ap + p * a_panel, &tm_x, x, 0, &sh.full[s]);
            tma_load_2d(bp + p * b_panel, &tm_w, x, col0, &sh.full[s]);
          }
        }
      } else {                               // the rank-r step: S_HL rows, U operand rows
        if (!wait_s_rows(a.flags, a.n_s, a.wait_epoch, abort, a.wait_cycles)) {
          ok = false;
          break;
        }
        fence_async_global();
        // r <= 32: one panel [hi | lo | 0]; r = 64: the hi and the lo panel
        constexpr int kP = R <= 32 ? 1 : 2;
        mbar_arrive_expect_tx(&sh.full[s], (uint32_t)(kP * (a_panel + b_panel)));
#pragma unroll
        for (int p = 0; p < kP; ++p) {
          tma_load_2d(ap + p * a_panel, &tm_s, 64 * p, 0, &sh.full[s]);
          tma_load_2d(bp + p * b_panel, &tm_u, 64 * p, a.u_row0 + col0, &sh.full[s]);
        }
      }
      ++n_st;
      if (++s == S) { s = 0; ph ^= 1u; }
    }
    if (!ok) {
      atomicOr(a.status, (uint32_t)kDevTimeout);
      *reinterpret_cast<volatile int*>(&sh.abort_flag) = 1;
    }
    // every copy has landed before this CTA leaves its shared memory
    for (int q = 0; q < S; ++q) {
      const int64_t last = last_in_slot(n_st, q, S);
      if (last >= 0) mbar_wait_bounded(&sh.full[q], (uint32_t)((last / S) & 1), nullptr, a.wait_cycles);
    }
  } else if (warp == 1 && lane == 0) {
    // ---------------------------------------------------------------- MMA issuer
    const uint32_t idesc = idesc_bf16_f32(128, b_rows);
    const uint64_t pa = (uint64_t)(a_panel >> 4), pb = (uint64_t)(b_panel >> 4);
    constexpr uint64_t kStepK = 32 >> 4;
    int s = 0;
    uint32_t ph = 0;
    for (int k = 0; k < n_k; ++k) {
      if (!mbar_wait_bounded(&sh.full[s], ph, abort, a.wait_cycles)) {
        atomicOr(a.status, (uint32_t)kDevTimeout);
        *reinterpret_cast<volatile int*>(&sh.abort_flag) = 1;
        break;
      }
      const uint64_t a0 = sdesc_k_sw128(smem_u32(smem + s * sbytes));
      const uint64_t b0 = sdesc_k_sw128(smem_u32(smem + s * sbytes + panels * a_panel));
      if (k < k_stages) {
        const int np = min(panels, a.k_steps - panels * k);
        for (int p = 0; p < np; ++p)
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
            mma_f16(tmem, a0 + p * pa + kk * kStepK, b0 + p * pb + kk * kStepK, idesc,
                    (k > 0 || p > 0 || kk > 0) ? 1u : 0u);
      } else if constexpr (R <= 32) {
        // hi chunk kk at element 16 kk of an operand row, lo chunk at R + 16 kk
#pragma unroll
        for (int kk = 0; kk < R / 16; ++kk) {
          const uint64_t hi = kk * kStepK, lo = (R / 16 + kk) * kStepK;
          mma_f16(tmem, a0 + hi, b0 + hi, idesc, 1u);
          mma_f16(tmem, a0 + hi, b0 + lo, idesc, 1u);
          mma_f16(tmem, a0 + lo, b0 + hi, idesc, 1u);
        }
      } else {
#pragma unroll
        for (int kk = 0; kk < 4; ++kk) {
          const uint64_t st = kk * kStepK;
          mma_f16(tmem, a0 + st, b0 + st, idesc, 1u);
          mma_f16(tmem, a0 + st, b0 + pb + st, idesc, 1u);
          mma_f16(tmem, a0 + pa + st, b0 + st, idesc, 1u);
        }
      }
      mma_commit(&sh.empty[s]);
      if (++s == S) { s = 0; ph ^= 1u; }
    }
    mma_commit(&sh.acc_full);              // after every MMA issued, a cut-short run's too
  }
  __syncwarp();
  if (!mbar_wait_bounded(&sh.acc_full, 0u, nullptr, a.wait_cycles))
    atomicOr(a.status, (uint32_t)kDevTimeout);
  tc_fence_after();

  const int g = warp & 3;                  // TMEM lanes 32 g .. + 31: tokens
  const uint32_t t_lane = tmem + ((uint32_t)(32 * g) << 16);
  if (is_s) {
    if (warp == 0) {
      // S's columns kSC s_blk .. for this lane's token: the sums of the P_hi and P_lo products
      const int row = s_tok + lane;
      uint32_t v[32], w[32];
      tmem_ld_32x32b_x32(t_lane, v);
      if constexpr (kSC == 32) tmem_ld_32x32b_x32(t_lane + 32, w);
      tmem_ld_wait();
      float x[kSC];
#pragma unroll
      for (int q = 0; q < kSC; ++q)
        x[q] = 0.f + (__uint_as_float(v[q]) + __uint_as_float(kSC == 32 ? w[q] : v[(16 + q) & 31]));
      if (row < a.T) {
        write_s_chunk<R>(a.s_hl, row, s_blk, x);
        if (s_blk == 0) zero_s_pad<R>(a.s_hl, row);
      }
      fence_async_global();
      __threadfence();
      __syncwarp();
      if (lane == 0) set_ready(a.flags + blockIdx.x, a.epoch);
    }
  } else if (32 * g < a.tokens) {
    const int row = 32 * g + lane;
    __nv_bfloat16* y = a.Y + (int64_t)row * a.ldy + col0;
    for (int c = 16 * (warp >> 2); c < a.cols; c += 32) {
      uint32_t v[16];
      tmem_ld_32x32b_x16(t_lane + c, v);
      tmem_ld_wait();
      uint32_t w[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const __nv_bfloat162 b2 =
            __floats2bfloat162_rn(__uint_as_float(v[2 * q]), __uint_as_float(v[2 * q + 1]));
        w[q] = *reinterpret_cast<const uint32_t*>(&b2);
      }
      // (m is a multiple of 8, and Y's rows are 16-byte aligned)
#pragma unroll
      for (int h = 0; h < 2; ++h)
        if (row < a.T && col0 + c + 8 * h < a.m)
          *reinterpret_cast<uint4*>(y + c + 8 * h) =
              make_uint4(w[4 * h], w[4 * h + 1], w[4 * h + 2], w[4 * h + 3]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

template <int R>
cudaError_t launch_few_r(const CUtensorMap& tm_x, const CUtensorMap& tm_xs, const CUtensorMap& tm_w,
                         const CUtensorMap& tm_pk, const CUtensorMap& tm_s, const CUtensorMap& tm_u,
                         const FewArgs& args, int ctas, size_t smem, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(linear_few_kernel<R>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  return launch_dependent(linear_few_kernel<R>, (unsigned)ctas, kThreads, smem, s, 1, true, tm_x, tm_xs,
                          tm_w, tm_pk, tm_s, tm_u, args);
}

int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

}  // namespace

LinearFewPlan linear_few_plan(int64_t T, int64_t m, int64_t n, int32_t r, int32_t sms) {
  LinearFewPlan pl{};
  if (T < 1 || T > kMaxTokens || m < 1 || n < 1 || (r != 16 && r != 32 && r != 64))
    return pl;
  pl.tokens = (int32_t)(ceil_div(T, 16) * 16);
  pl.s_cols = s_cols(r);
  pl.s_tokens = kSTokens;
  pl.n_s = (int32_t)(ceil_div(T, kSTokens) * (r / pl.s_cols));
  // one wave of CTAs beside those of S, on all the SMs
  const int64_t free_sms = std::max<int64_t>(1, sms - pl.n_s);
  pl.cols = (int32_t)std::min<int64_t>(128, ceil_div(ceil_div(m, free_sms), 16) * 16);
  // the SM-pair kernel takes what needs more than one wave
  if (ceil_div(m, pl.cols) > free_sms) return LinearFewPlan{};
  pl.ctas = (int32_t)(pl.n_s + ceil_div(m, pl.cols));
  const int64_t budget = 208 * 1024 - kASpan;
  const int64_t panel = 128 * (int64_t)(pl.tokens + pl.cols);
  const int64_t s_panel = 128 * (int64_t)(kSTokens + 2 * pl.s_cols);
  // stages of as many panels as leave three of them: each stage's wait and commit costs the
  // MMAs some 300 cycles (4096 x 4096 at 97 tokens: 19.0 us with two panels and five stages,
  // 17.3 with three and three), but two stages no longer cover the loads (4096 x 11008 at 97
  // tokens: 39 us against 37)
  constexpr int kTargetStages = 3;
  pl.panels = (int32_t)std::min<int64_t>(8, std::max<int64_t>(2, budget / kTargetStages / panel));
  pl.s_panels = (int32_t)std::min<int64_t>(8, std::max<int64_t>(2, budget / kTargetStages / s_panel));
  const int64_t st = pl.panels * panel, s_st = pl.s_panels * s_panel;
  pl.stages = (int32_t)std::min<int64_t>(kMaxStages, budget / st);
  pl.s_stages = (int32_t)std::min<int64_t>(kMaxStages, budget / s_st);
  // an MMA reads kASpan bytes from each panel of A on, in the last stage past its end
  pl.smem = std::max(pl.stages * st, pl.s_stages * s_st) + kASpan + 1024;
  return pl;
}

cudaError_t launch_linear_few(const CUtensorMap& tm_x, const CUtensorMap& tm_xs,
                              const CUtensorMap& tm_w, const CUtensorMap& tm_pk,
                              const CUtensorMap& tm_s, const CUtensorMap& tm_u,
                              const LinearFewPlan& plan, int64_t T, int64_t m, int64_t n, int32_t r,
                              int32_t u_row0, __nv_bfloat16* s_hl, uint32_t* flags, uint32_t epoch,
                              __nv_bfloat16* Y, int64_t ldy, bool inject_wait, uint32_t* d_status,
                              cudaStream_t s) {
  if (plan.ctas < 1 || plan.stages < 2 || plan.s_stages < 2 || plan.stages > kMaxStages ||
      plan.s_stages > kMaxStages || plan.n_s > kLinearFewFlags || plan.cols < 16 || plan.cols > 128)
    return cudaErrorInvalidValue;
  FewArgs a{};
  a.T = (int)T;
  a.m = (int)m;
  a.tokens = plan.tokens;
  a.cols = plan.cols;
  a.k_steps = (int)ceil_div(n, 64);
  a.n_s = plan.n_s;
  a.panels = plan.panels;
  a.s_panels = plan.s_panels;
  a.stages = plan.stages;
  a.s_stages = plan.s_stages;
  a.u_row0 = u_row0;
  a.ldy = ldy;
  a.Y = Y;
  a.s_hl = s_hl;
  a.flags = flags;
  a.epoch = epoch;
  a.wait_epoch = inject_wait ? epoch + 1 : epoch;
  a.status = d_status;
  a.wait_cycles = inject_wait ? kTestWaitCycles : kWaitCycles;
#define ZO_FEW(RR)                                                                               \
  case RR:                                                                                       \
    return launch_few_r<RR>(tm_x, tm_xs, tm_w, tm_pk, tm_s, tm_u, a, plan.ctas, (size_t)plan.smem, s)
  switch (r) {
    ZO_FEW(16);
    ZO_FEW(32);
    ZO_FEW(64);
    default: return cudaErrorInvalidValue;
  }
#undef ZO_FEW
}

}  // namespace zo
