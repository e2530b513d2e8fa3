// Device-side definitions shared by the kernels of the SubZero+ weight path.
//
// The random-number contract (Philox4x32-10 + uniform + Box-Muller) is written
// here from its published definitions (Salmon et al., SC'11; Box & Muller 1958)
// and is the only source of Z_i^(k) (Sec. 4.1, Eq. (4); App. A.1 seed trick) and
// of Omega_U / Omega_V (Alg. 1) on the GPU.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>
#include <cuda_bf16.h>

namespace zo {

// ---------------------------------------------------------------------------
// Status words written by kernels (read back by zo_sync_status).
// ---------------------------------------------------------------------------
enum DeviceStatus : uint32_t {
  kDevOk = 0,
  kDevTimeout = 1,   // a bounded mbarrier / flag wait gave up
  kDevBounds = 2,    // an internal bound check failed; the access was skipped
  kDevNotPosDef = 4, // refresh: a Gram matrix had a non-positive Cholesky pivot
};

// Two fp32 operations (each lane rounded to nearest, as fmaf and *) in one instruction.
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, c, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\tmov.b64 c, {%6, %7};\n\t"
      "fma.rn.f32x2 d, a, b, c;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y), "f"(c.x), "f"(c.y));
  return d;
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  float2 d;
  asm("{\n\t.reg .b64 a, b, d;\n\t"
      "mov.b64 a, {%2, %3};\n\tmov.b64 b, {%4, %5};\n\t"
      "mul.rn.f32x2 d, a, b;\n\tmov.b64 {%0, %1}, d;\n\t}"
      : "=f"(d.x), "=f"(d.y)
      : "f"(a.x), "f"(a.y), "f"(b.x), "f"(b.y));
  return d;
}

// ---------------------------------------------------------------------------
// Counter contract
// ---------------------------------------------------------------------------
constexpr uint32_t kTagZ = 1;
constexpr uint32_t kTagOmegaU = 2;
constexpr uint32_t kTagOmegaV = 3;

__host__ __device__ constexpr uint32_t query_word(uint32_t tag, uint32_t k) {
  return (tag << 24) | (k & 0xFFFFFFu);
}

// Philox4x32 with ten rounds.  Round: (x0,x1,x2,x3) -> (hi(B*x2)^x1^k0, lo(B*x2),
// hi(A*x0)^x3^k1, lo(A*x0)) with A = 0xD2511F53, B = 0xCD9E8D57; the key is
// advanced by the Weyl constants (0x9E3779B9, 0xBB67AE85) between rounds.
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int rnd = 0; rnd < 10; ++rnd) {
    if (rnd > 0) {
      k0 += 0x9E3779B9u;
      k1 += 0xBB67AE85u;
    }
    const uint64_t a = (uint64_t)0xD2511F53u * c.x, b = (uint64_t)0xCD9E8D57u * c.z;
    const uint32_t hi_a = (uint32_t)(a >> 32), lo_a = (uint32_t)a;
    const uint32_t hi_b = (uint32_t)(b >> 32), lo_b = (uint32_t)b;
    c = make_uint4(hi_b ^ c.y ^ k0, lo_b, hi_a ^ c.w ^ k1, lo_a);
  }
  return c;
}

// u = ((x >> 8) + 1) * 2^-24 in (0, 1]; the integer fits 24 bits, so exact in fp32.
__device__ __forceinline__ float u01(uint32_t x) {
  return __uint2float_rn((x >> 8) + 1u) * 5.9604644775390625e-08f;
}

// Box-Muller on kV vectors of word pairs (xa, xb), u = ((x >> 8) + 1) 2^-24 in (0, 1]:
// rad cos 2 pi ub = nr c and rad sin 2 pi ub = nr s with nr = -rad = -sqrt(-2 ln ua).  The
// uniforms are integers over 2^24, so both functions reduce their arguments exactly, in
// integers:
//  * ln: k = u 2^24 = m 2^e with m near 1 (the reduction of Cody and Waite, Software Manual for
//    the Elementary Functions, 1980), in [2/3, 4/3), where m - 1 reaches as far to either side:
//    k's bits less those of (2/3) 2^24 hold e - 24 above the mantissa.  g = 2 m - 2 exact,
//    2 ln u = (e - 24) 2 ln 2 + g + g^2 P(g), P of degree 8.
//  * sqrt of x = -2 ln u: the hardware's reciprocal square root y, s = x y, and one Newton
//    step by the residual, s + (x - s^2) y / 2 (Markstein, IBM J. Res. Dev. 34, 1990), all with
//    the sign turned; u = 1 gives 0.
//  * cos, sin: k + 2^21 = quadrant 2^22 + j, the angle inside the quadrant (pi/4) t with
//    t = (j - 2^21) 2^-21 exact in [-1, 1); sin = t s0 + t q(t^2) with s0 the fp32 pi/4 and
//    its error in q, cos = 1 + t^2 p(t^2), q and p of degree 3; the quadrant swaps and negates.
// The polynomials are minimax fits to the functions (made again in
// tests/test_packed_normal_fit.py): P for the relative error with P(0) given, and q, rounded to
// fp32 from the lowest order on, the rest fitted again; p rounded at once.  Their errors: ln
// 5.8e-9 of the result, sin 2.5e-9, cos 8.7e-9.
// Over all 2^24 uniforms (double precision): radius within 3.5e-7 (rms 4.05e-8), cos and sin
// within 6.1e-8, no further off than logf, sqrtf and sincospif.
template <int kV>
__device__ __forceinline__ void box_muller_parts(const uint32_t (&xa)[2 * kV],
                                                 const uint32_t (&xb)[2 * kV], float2 (&nr)[kV],
                                                 float2 (&zc)[kV], float2 (&zs)[kV]) {
  auto all = [](float x) { return make_float2(x, x); };
  {
    float2 g[kV], e[kV], P[kV];
#pragma unroll
    for (int v = 0; v < kV; ++v) {
      float m[2], x[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) {
        const int k = __float_as_int(__uint2float_rn((xa[v * 2 + l] >> 8) + 1u));
        const int ex = (k - 0x4b2aaaab) & (int)0xff800000;     // (e - 24) 2^23
        m[l] = __int_as_float(k - ex - 0x0c000000);
        x[l] = __int2float_rn(ex);
      }
      g[v] = fma2(make_float2(m[0], m[1]), all(2.0f), all(-2.0f));
      e[v] = make_float2(x[0], x[1]);
    }
    constexpr float kP[9] = {-0x1p-2f,        0x1.55550cp-4f,  -0x1.fffe5ep-6f,
                             0x1.99ce34p-7f,  -0x1.55b7ecp-8f, 0x1.1ef264p-9f,
                             -0x1.f03bdcp-11f, 0x1.1defc4p-11f, -0x1.0e2acep-12f};
#pragma unroll
    for (int v = 0; v < kV; ++v) P[v] = all(kP[8]);
#pragma unroll
    for (int i = 7; i >= 0; --i)
#pragma unroll
      for (int v = 0; v < kV; ++v) P[v] = fma2(P[v], g[v], all(kP[i]));
#pragma unroll
    for (int v = 0; v < kV; ++v) {
      float2 nl = fma2(mul2(g[v], g[v]), P[v], g[v]);
      nl = fma2(e[v], all(0x1.62e430p-23f), nl);               // 2 ln u
      float2 y;
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.x) : "f"(fmaxf(-nl.x, 1e-30f)));
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y.y) : "f"(fmaxf(-nl.y, 1e-30f)));
      const float2 ns = mul2(nl, y);
      nr[v] = fma2(fma2(ns, ns, nl), mul2(y, all(0.5f)), ns);
    }
  }
  uint32_t qd[2 * kV];                                         // (k + 2^21) 2^8
  float2 t[kV], w[kV], sn[kV], cs[kV];
#pragma unroll
  for (int v = 0; v < kV; ++v) {
    float j[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      qd[v * 2 + l] = xb[v * 2 + l] + 0x20000100u;
      j[l] = __uint_as_float(((qd[v * 2 + l] >> 8) & 0x3fffffu) | 0x4b000000u);   // 2^23 + j
    }
    t[v] = fma2(make_float2(j[0], j[1]), all(0x1p-21f), all(-5.0f));
    w[v] = mul2(t[v], t[v]);
  }
  constexpr float kS[4] = {-0x1.a0f38ap-26f, -0x1.4abbbap-4f, 0x1.465ee8p-9f, -0x1.2da132p-15f};
  constexpr float kC[4] = {-0x1.3bd3ccp-2f, 0x1.03c1e2p-6f, -0x1.55c752p-12f, 0x1.da30fap-19f};
#pragma unroll
  for (int v = 0; v < kV; ++v) { sn[v] = all(kS[3]); cs[v] = all(kC[3]); }
#pragma unroll
  for (int i = 2; i >= 0; --i)
#pragma unroll
    for (int v = 0; v < kV; ++v) {
      sn[v] = fma2(w[v], sn[v], all(kS[i]));
      cs[v] = fma2(w[v], cs[v], all(kC[i]));
    }
#pragma unroll
  for (int v = 0; v < kV; ++v) {
    sn[v] = fma2(t[v], all(0x1.921fb6p-1f), mul2(t[v], sn[v]));
    cs[v] = fma2(w[v], cs[v], all(1.0f));
    const float a[2] = {cs[v].x, cs[v].y}, b[2] = {sn[v].x, sn[v].y};
    float c[2], s[2];
#pragma unroll
    for (int l = 0; l < 2; ++l) {
      const uint32_t q = qd[v * 2 + l];
      const bool odd = (q & 0x40000000u) != 0;
      // cos is negative in quadrants 1 and 2, sin in 2 and 3; both negated, as nr is -rad
      c[l] = __uint_as_float(__float_as_uint(odd ? b[l] : a[l]) ^ ((q + 0xc0000000u) & 0x80000000u));
      s[l] = __uint_as_float(__float_as_uint(odd ? a[l] : b[l]) ^ (~q & 0x80000000u));
    }
    zc[v] = make_float2(c[0], c[1]);
    zs[v] = make_float2(s[0], s[1]);
  }
}

// The same of one pair of words by CUDA's functions: what forms Z, and Omega but for the panels
// of fp32 weights at r = 4 and 8 with 4 r rows or more that clusters hold in registers
// (zo_cholqr_small.cu; those and the full-space pass take the transform above).  The two differ in the last
// place, and bf16 weights at a rounding boundary show it: up to rel 1.3e-5 of a 1 M-weight set
// after a step.
__device__ __forceinline__ float2 box_muller(uint32_t xa, uint32_t xb) {
  const float rad = sqrtf(-2.0f * logf(u01(xa)));
  float s, c;
  sincospif(2.0f * u01(xb), &s, &c);
  return make_float2(rad * c, rad * s);
}

// Four normals of counter word `c4` of the stream (seed, x1, x2, x3).
__device__ __forceinline__ float4 normal4(uint64_t seed, uint32_t c4, uint32_t x1, uint32_t x2,
                                          uint32_t x3) {
  const uint4 w = philox4x32_10(make_uint4(c4, x1, x2, x3), static_cast<uint32_t>(seed),
                                static_cast<uint32_t>(seed >> 32));
  const float2 a = box_muller(w.x, w.y);
  const float2 b = box_muller(w.z, w.w);
  return make_float4(a.x, a.y, b.x, b.y);
}
__device__ __forceinline__ float4 normal4_packed(uint64_t seed, uint32_t c4, uint32_t x1,
                                                 uint32_t x2, uint32_t x3) {
  const uint4 w = philox4x32_10(make_uint4(c4, x1, x2, x3), static_cast<uint32_t>(seed),
                                static_cast<uint32_t>(seed >> 32));
  const uint32_t a[2] = {w.x, w.z}, b[2] = {w.y, w.w};
  float2 nr[1], c[1], s[1];
  box_muller_parts<1>(a, b, nr, c, s);
  c[0] = mul2(nr[0], c[0]);
  s[0] = mul2(nr[0], s[0]);
  return make_float4(c[0].x, s[0].x, c[0].y, s[0].y);
}

// ---------------------------------------------------------------------------
// Matrix descriptor as seen by the kernels (built by the host runtime).
// ---------------------------------------------------------------------------
struct MatDesc {
  void* W;          // m x n, leading dimension ldw (elements)
  int64_t m, n, ldw;
  int32_t dtype;    // 0 = fp32, 1 = bf16
  uint32_t gidx;    // global Philox matrix index
  float* U;         // m x r
  float* V;         // n x r
  float* M;         // r x r first moment
  float* Vm;        // r x r second moment
  float* C;         // r x r coefficient of the current pass (workspace)
  float* P;         // FMA path: r x n, P = C V^T (workspace)
  int64_t tile0;    // first 32-row tile of this matrix (one-launch FMA passes, MeZO)
};

// Per-matrix record of the tensor-core weight pass (128 x 128 tiles).
struct TcMat {
  int64_t m, n;
  int64_t tile0;     // first tile of this matrix
  int32_t tiles_n;   // column tiles
  int32_t u_row0;    // first row of this matrix in the stacked hi/lo U operand
  int32_t p_row0;    // first row of this matrix in the stacked hi/lo P^T operand
  int32_t pad;
};

// One block of the batched TSQR used by the refresh (see zo_qr.cu).
struct QrBlock {
  float* rows;         // storage of this block's rows (R floats per row)
  const float* s_in;   // down pass: the R x R block of the parent's Q for this block
  float* r_out;        // up pass: where this block's R x R triangular factor goes
  float* tau;          // R Householder scalars of this block
  int64_t row0;        // level 0: first panel row of the block (element addressing of Omega)
  int32_t n_real;      // rows of real data in the block (the rest is zero padding)
  int32_t flags;       // kQrTop | kQrLevel0
  uint32_t gidx;       // matrix index for Omega
  uint32_t tag;        // kTagOmegaU or kTagOmegaV
};
constexpr int32_t kQrTop = 1;
constexpr int32_t kQrLevel0 = 2;

}  // namespace zo
