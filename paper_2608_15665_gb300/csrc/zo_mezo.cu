// Full-space SPSA perturbation of MeZO, Eq. (1): W_i <- rnd(W_i + coef * Z_i) with
// Z_i[row, col] ~ N(0, 1) drawn per element from the counter contract:
//   counter = (row * ceil(n_i / 4) + col / 4, matrix index, t, 5 << 24), lane col % 4.
// coef = +eps / -2 eps / +eps gives the two evaluations of Eq. (1) and the restore;
// coef = eps - eta * rho fuses the restore with MeZO's SGD update.
//
// Unlike the subspace pass, every weight needs its own Gaussian: one Philox4x32-10
// call and two Box-Muller transforms per 4 weights, so the pass is bound by the ALU
// (integer multiplies, log / sqrt / sincos), not by HBM: 38 thread instructions per weight
// and 8.73 ms a pass on the 7B set (59 and 12.2 with CUDA's log and sincos).  Tiles are
// 32 rows x (32 lanes x 16 bytes): a warp reads and writes 512 contiguous bytes of a row,
// each thread draws the 2 (bf16) or 1 (fp32) counter words of its 16 bytes.
#include "zo_fma_common.cuh"

namespace zo {
namespace {

using namespace fma;

constexpr uint32_t kTagMezo = 5;

// The Philox round keys of one seed: (k0, k1) = (seed_lo, seed_hi) advanced by the Weyl
// constants (0x9E3779B9, 0xBB67AE85) once per round -- the key schedule of zo_device.cuh's
// philox4x32_10, formed once on the host.  Passed as a kernel parameter, each key is read
// from the constant bank by the round's XOR: the eight Philox calls of a thread spend no
// instructions and no registers on it.
struct RoundKeys {
  uint32_t k0[10], k1[10];
};

RoundKeys round_keys(uint64_t seed) {
  RoundKeys k;
  k.k0[0] = (uint32_t)seed;
  k.k1[0] = (uint32_t)(seed >> 32);
  for (int r = 1; r < 10; ++r) {
    k.k0[r] = k.k0[r - 1] + 0x9E3779B9u;
    k.k1[r] = k.k1[r - 1] + 0xBB67AE85u;
  }
  return k;
}

// philox4x32_10 of zo_device.cuh with the round keys given.
__device__ __forceinline__ uint4 philox_keyed(const RoundKeys& k, uint4 c) {
#pragma unroll
  for (int rnd = 0; rnd < 10; ++rnd) {
    const uint64_t a = (uint64_t)0xD2511F53u * c.x, b = (uint64_t)0xCD9E8D57u * c.z;
    const uint32_t hi_a = (uint32_t)(a >> 32), lo_a = (uint32_t)a;
    const uint32_t hi_b = (uint32_t)(b >> 32), lo_b = (uint32_t)b;
    c = make_uint4(hi_b ^ c.y ^ k.k0[rnd], lo_b, hi_a ^ c.w ^ k.k1[rnd], lo_a);
  }
  return c;
}

// One tile's rows of this thread's 16 bytes, kRows at a time, their counters' normals formed
// together in packed arithmetic.  Bound by the FMA pipe (80% busy on 201 M bf16 weights:
// 18 wide multiplies of the Philox rounds and some 35 packed operations per counter, 145
// instructions where the precise logf / sqrtf / sincospif took 238) and by issue (69%):
// 275 us against 379 us, 1.4 ps per weight; two counters at a time (one row of bf16, two of
// fp32), as four measured 317 us, and 32 registers for eight CTAs per SM (six: 4% slower).
template <typename T, int kRows>
__device__ __forceinline__ void mezo_tile(const MatDesc& md, int64_t local, const RoundKeys& keys,
                                          uint32_t t, float coef) {
  constexpr int VEC = Vec<T>::N, kCtr = VEC / 4;      // elements, counters per row
  constexpr int64_t TN = 32 * VEC;
  const int64_t tiles_n = (md.n + TN - 1) / TN;
  const int64_t row0 = (local / tiles_n) * kFmaTileRows;
  const int64_t col = (local % tiles_n) * TN + (threadIdx.x & 31) * VEC;
  if (col >= md.n) return;
  const uint32_t n4 = (uint32_t)((md.n + 3) / 4);
  const uint32_t x3 = query_word(kTagMezo, 0);
  const bool full = col + VEC <= md.n;
  T* W = reinterpret_cast<T*>(md.W) + col;
#pragma unroll 1
  for (int rr = threadIdx.x >> 5; rr < kFmaTileRows; rr += 8 * kRows) {
    if (row0 + rr >= md.m) break;
    uint4 raw[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      raw[i] = make_uint4(0u, 0u, 0u, 0u);
      const int64_t row = row0 + rr + 8 * i;
      if (full && row < md.m) raw[i] = *reinterpret_cast<const uint4*>(W + row * md.ldw);
    }
    constexpr int kN = 2 * kCtr * kRows;               // pairs
    uint32_t xa[kN], xb[kN];
#pragma unroll
    for (int i = 0; i < kRows; ++i)
#pragma unroll
      for (int c = 0; c < kCtr; ++c) {
        const uint32_t c4 = (uint32_t)((row0 + rr + 8 * i) * n4 + col / 4) + c;
        const uint4 x = philox_keyed(keys, make_uint4(c4, md.gidx, t, x3));
        const int p = 2 * (i * kCtr + c);
        xa[p] = x.x; xb[p] = x.y; xa[p + 1] = x.z; xb[p + 1] = x.w;
      }
    float2 nr[kN / 2], zc[kN / 2], zs[kN / 2];
    box_muller_parts<kN / 2>(xa, xb, nr, zc, zs);
#pragma unroll
    for (int p = 0; p < kN / 2; ++p) {
      zc[p] = mul2(nr[p], zc[p]);
      zs[p] = mul2(nr[p], zs[p]);
    }
    const float2 coef2 = make_float2(coef, coef);
#pragma unroll
    for (int i = 0; i < kRows; ++i) {
      const int64_t row = row0 + rr + 8 * i;
      if (row >= md.m) break;
      T* w = W + row * md.ldw;
      if (full) {
        const uint32_t v[4] = {raw[i].x, raw[i].y, raw[i].z, raw[i].w};
        uint32_t o[4];
#pragma unroll
        for (int c = 0; c < kCtr; ++c) {
          const int p = i * kCtr + c;
          // elements 0, 2 of the counter take the cosines, 1, 3 the sines
          float2 even, odd;
          if constexpr (VEC == 8) {
            even = make_float2(__uint_as_float(v[2 * c] << 16), __uint_as_float(v[2 * c + 1] << 16));
            odd = make_float2(__uint_as_float(v[2 * c] & 0xFFFF0000u),
                              __uint_as_float(v[2 * c + 1] & 0xFFFF0000u));
          } else {
            even = make_float2(__uint_as_float(v[0]), __uint_as_float(v[2]));
            odd = make_float2(__uint_as_float(v[1]), __uint_as_float(v[3]));
          }
          even = fma2(coef2, zc[p], even);
          odd = fma2(coef2, zs[p], odd);
          if constexpr (VEC == 8) {
            o[2 * c] = pack2_bf16(even.x, odd.x);
            o[2 * c + 1] = pack2_bf16(even.y, odd.y);
          } else {
            o[0] = __float_as_uint(even.x); o[1] = __float_as_uint(odd.x);
            o[2] = __float_as_uint(even.y); o[3] = __float_as_uint(odd.y);
          }
        }
        *reinterpret_cast<uint4*>(w) = make_uint4(o[0], o[1], o[2], o[3]);
      } else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) {
          const int p = i * kCtr + k / 4;
          const float2 z = k & 1 ? zs[p] : zc[p];
          if (col + k < md.n)
            store_scalar<T>(w + k, fmaf(coef, k & 2 ? z.y : z.x, load_scalar<T>(w + k)));
        }
      }
    }
  }
}

__global__ void __launch_bounds__(256, 8)
mezo_kernel(const MatDesc* __restrict__ mats, int n_mats, const int64_t* __restrict__ prefix,
            const __grid_constant__ RoundKeys keys, uint32_t t, float coef) {
  const int64_t tile = blockIdx.x;
  const MatDesc md = mats[find_matrix(prefix, n_mats, tile)];
  const int64_t local = tile - md.tile0;
  if (md.dtype == 1)
    mezo_tile<__nv_bfloat16, 1>(md, local, keys, t, coef);
  else
    mezo_tile<float, 2>(md, local, keys, t, coef);
}

}  // namespace

cudaError_t launch_mezo(const MatDesc* d_mats, int32_t n_mats, const int64_t* d_tile_prefix,
                        int64_t n_tiles, uint64_t seed, uint32_t t, float coef, cudaStream_t s) {
  if (n_tiles <= 0) return cudaSuccess;
  if (n_tiles > 0x7FFFFFFF) return cudaErrorInvalidValue;
  mezo_kernel<<<(unsigned)n_tiles, 256, 0, s>>>(d_mats, n_mats, d_tile_prefix, round_keys(seed), t,
                                                coef);
  return cudaGetLastError();
}

}  // namespace zo
