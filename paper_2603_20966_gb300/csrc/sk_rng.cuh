// sk_rng.cuh -- device-side generator of the sketching matrix entries.
//
// Entry (r, c) of the generated matrix is a pure function of
// (seed, r, c): any CTA that needs it regenerates it instead of reading it,
// which is the single-GPU form of the paper's choice to generate the random
// matrix redundantly on every processor rather than communicate it
// (arXiv 2603.20966, Sec. 6.2, "Communicate vs Redundantly Generate Omega",
// Philox with a shared seed; Alg. 1 GenRandom).
//
// Specification (identical bit for bit to the CPU oracle, written
// independently here):
//   key      = (seed lo32, seed hi32)
//   counter  = (c >> 2, r, dom, 0) for Gaussian/uniform (4 entries per call),
//              (c >> 7, r, dom, 0) for Rademacher (128 entries per call)
//   Philox4x32-10 (Salmon et al., SC'11): 10 rounds, multipliers
//   0xD2511F53 / 0xCD9E8D57, Weyl key increments 0x9E3779B9 / 0xBB67AE85.
//   Gaussian: Box-Muller on (x0,x1) for c%4 in {0,1}, (x2,x3) for {2,3}:
//     u1 = ((xa>>8)+1) 2^-24, rho = sqrt(-2 ln u1); from xb the position
//     r = (bits 29..8) 2^-23 - 1/4 and (X, Y) = (cospi r, sinpi r) turned by
//     q = bits 31..30 quarter turns (angle pi r + q pi/2: the 2^24 words give
//     every multiple of 2 pi / 2^24 once); g = rho X (c even) or rho Y (c odd).
//   Rademacher: bit c%32 of word (c>>5)%4, set -> -1.
//   Uniform: (x_{c%4} >> 8) 2^-24.
// Every floating-point step is an explicitly rounded IEEE operation
// (__fadd2_rn, __fmul2_rn, __ffma2_rn and their scalar forms), so no
// compiler contraction or fast-math flag can change a bit.  ln, sin and cos
// are polynomials; the square root of Box-Muller is the correctly rounded
// IEEE result, computed by Markstein's method from the hardware
// reciprocal-square-root approximation (see neg_sqrt_neg_x2).
#pragma once
#include <stdint.h>
#include <cuda_bf16.h>
#include <cuda_fp8.h>

namespace sk {

enum : int { kGaussian = 0, kRademacher = 1, kUniform = 2 };
enum : int { kFP32 = 0, kBF16 = 1, kE4M3 = 2 };

struct PhiloxKey {
  uint32_t k0, k1;
};

__host__ __device__ inline PhiloxKey make_key(uint64_t seed) {
  return PhiloxKey{(uint32_t)(seed & 0xffffffffu), (uint32_t)(seed >> 32)};
}

// The key words of all ten rounds, (k0 + i 0x9E3779B9, k1 + i 0xBB67AE85) at
// k[2i], k[2i+1].  A kernel that receives them among its launch parameters
// reads each one as a constant operand of the round's XOR instead of
// stepping the key in registers on every call.
struct PhiloxRoundKeys {
  uint32_t k[20];
};

__host__ __device__ inline PhiloxRoundKeys round_keys(PhiloxKey key) {
  PhiloxRoundKeys rk;
  for (int i = 0; i < 10; ++i) {
    rk.k[2 * i] = key.k0 + (uint32_t)i * 0x9E3779B9u;
    rk.k[2 * i + 1] = key.k1 + (uint32_t)i * 0xBB67AE85u;
  }
  return rk;
}

__device__ __forceinline__ uint32_t round_key(const PhiloxKey& key, int i, int w) {
  return w == 0 ? key.k0 + (uint32_t)i * 0x9E3779B9u : key.k1 + (uint32_t)i * 0xBB67AE85u;
}
__device__ __forceinline__ uint32_t round_key(const PhiloxRoundKeys& rk, int i, int w) {
  return rk.k[2 * i + w];
}

// Philox4x32-10 on the counter (j, r, 0, 0), K = PhiloxKey or PhiloxRoundKeys.
// With two counter words zero, one of the first three rounds' six products
// is zero and four depend on j alone or on r alone: PhiloxCol holds what entry
// column j contributes after round 3, PhiloxRow what row r does, and
// philox_join mixes one of each, with 15 wide products instead of 19 per
// call.  A wide product takes four cycles of the FMA pipe's multiply half
// (Philox alone, 19 of them per 4 entries, caps an SM at 6.3 entries per
// cycle), so threads that generate several entries of one row or one column
// keep its part.  Together with the shorter Box-Muller below (no operand
// negations, no refinement of the root, 5 packed operations fewer per 4
// entries): left 2^20 x 512, k = 2048 4.56 -> 4.39 ms, FP8 right 65536 x
// 16384, k = 256 1.477 -> 1.445 ms, batch of 256 5.21 -> 4.98 ms.
struct alignas(16) PhiloxCol {
  uint32_t a, b, c, d;
};
struct PhiloxRow {
  uint32_t h, l;
};

template <class K>
__device__ __forceinline__ PhiloxRow philox_row(const K& key, uint32_t r) {
  const uint32_t n0 = r ^ round_key(key, 0, 0);  // round 1 (its products by zero words drop out)
  return PhiloxRow{__umulhi(0xD2511F53u, n0), 0xD2511F53u * n0};  // round 2, word 0
}

template <class K>
__device__ __forceinline__ PhiloxCol philox_col(const K& key, uint32_t j) {
  const uint32_t lo0 = 0xD2511F53u * j;  // round 1, word 0
  const uint32_t n2 = __umulhi(0xD2511F53u, j) ^ round_key(key, 0, 1);
  const uint32_t c0 = __umulhi(0xCD9E8D57u, n2) ^ round_key(key, 1, 0);  // round 2, word 2
  const uint32_t c1 = 0xCD9E8D57u * n2;
  return PhiloxCol{lo0 ^ round_key(key, 1, 1), c1 ^ round_key(key, 2, 0),
                   __umulhi(0xD2511F53u, c0) ^ round_key(key, 2, 1),  // round 3, word 0
                   0xD2511F53u * c0};
}

template <class K>
__device__ __forceinline__ uint4 philox_join(const PhiloxRow& row, const PhiloxCol& col,
                                             const K& key) {
  const uint32_t x = row.h ^ col.a;  // word 2 after round 2
  uint32_t c0 = __umulhi(0xCD9E8D57u, x) ^ col.b;
  uint32_t c1 = 0xCD9E8D57u * x;
  uint32_t c2 = col.c ^ row.l;
  uint32_t c3 = col.d;
#pragma unroll
  for (int i = 3; i < 10; ++i) {
    const uint32_t lo0 = 0xD2511F53u * c0;
    const uint32_t hi0 = __umulhi(0xD2511F53u, c0);
    const uint32_t lo1 = 0xCD9E8D57u * c2;
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c2);
    c0 = hi1 ^ c1 ^ round_key(key, i, 0);
    c2 = hi0 ^ c3 ^ round_key(key, i, 1);
    c1 = lo1;
    c3 = lo0;
  }
  return make_uint4(c0, c1, c2, c3);
}

template <class K>
__device__ __forceinline__ uint4 philox(uint32_t j, uint32_t r, const K& key) {
  return philox_join(philox_row(key, r), philox_col(key, j), key);
}

// ---- Box-Muller on the two word pairs of one Philox call ----
// The two transforms run side by side: __fadd2_rn / __fmul2_rn / __ffma2_rn
// round each component exactly like the scalar __fadd_rn / __fmul_rn /
// __fmaf_rn, so every value is the one the specification's scalar steps give
// while the floating-point work takes half the instructions (the generator
// is instruction-issue bound inside the sketch kernels).  The square root
// gives the IEEE correctly rounded result (neg_sqrt_neg_x2).
// Where a step below is written differently from the specification, the
// comment beside it shows that the value is the same.
__device__ __forceinline__ float2 f2(float a, float b) { return make_float2(a, b); }

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// -sqrt(-u) with the root rounded to nearest-even, for u = 2 ln u1 in
// [-34, -2^-23] or u = +0 (u1 = 1, result +0).  Markstein's correction of
// w = -u from an approximate reciprocal square root y: g = w y, the exact
// residual d = w - g^2 (one FMA), g + d (y / 2), rounded once.  With this
// chip's approximation every one of the 2^24 radicands gives the IEEE root
// (test_gpu_box_muller_all runs them all); a seed a whole ulp from the
// rounded one would miss it for 3 of them, and a refinement of g and y / 2
// before the correction (three more FMAs) makes that up to 6 ulp none.
// Every step holds the negated values (u = -w, -g, -d), each the exact
// negative of the step above, so that no operand is negated by an
// instruction of its own.  The seed is taken at max(w, 1e-30), which changes
// nothing for w >= 2^-23 and keeps it finite at u = +0, where every step then
// yields +0.
__device__ __forceinline__ float2 neg_sqrt_neg_x2(float2 u) {
  const float2 y = f2(rsqrt_approx(fmaxf(-u.x, 1e-30f)), rsqrt_approx(fmaxf(-u.y, 1e-30f)));
  const float2 ng = __fmul2_rn(u, y);
  const float2 h = __fmul2_rn(f2(0.5f, 0.5f), y);
  const float2 nd = __ffma2_rn(ng, ng, u);
  return __ffma2_rn(nd, h, ng);
}

// 2 ln(x 2^-24) for integers x in [1, 2^24] given as floats: with
// x 2^-24 = 2^e f, f folded into [sqrt(1/2), sqrt 2), t = f - 1 (exact),
// ln f = t + t^2 Q(t) with Q of degree 8 (the generator specification's
// least-squares coefficients), ln x = e ln2_hi + (e ln2_lo + ln f).  The
// factors 2 are carried by the operands: w = 2t, the coefficient of t^i
// times 2^(-i - 1) (so that w^2 P(w) = 2 t^2 Q(t)), and 2 ln2_hi, 2 ln2_lo.  Scaling by powers of two commutes with rounding here, so every
// step is twice (or a power of two times) the specification's.
__device__ __forceinline__ float2 ln2x_x2(float2 x) {
  const uint32_t b0 = __float_as_uint(x.x), b1 = __float_as_uint(x.y);
  // Fold and split by one integer add: with m the mantissa bits, b + 0x4afb0c
  // carries into the exponent field exactly when m > 0x3504f3 (the fold), so
  // its exponent field is E (plus one when folded) and its mantissa field
  // plus 0x3f3504f4 is m with the exponent of 1 (or of 1/2 when folded).
  const uint32_t i0 = b0 + 0x004afb0cu, i1 = b1 + 0x004afb0cu;
  // e as a float without a conversion: 0x4B000000 + E is the float 2^23 + E
  // (E < 2^8), and subtracting 2^23 + 127 + 24 is exact
  const float2 eb = f2(__uint_as_float(0x4B000000u + (i0 >> 23)),
                       __uint_as_float(0x4B000000u + (i1 >> 23)));
  const float2 ef = __fadd2_rn(eb, f2(-8388759.0f, -8388759.0f));
  const float2 f = f2(__uint_as_float((i0 & 0x007fffffu) + 0x3f3504f4u),
                      __uint_as_float((i1 & 0x007fffffu) + 0x3f3504f4u));
  const float2 w = __ffma2_rn(f, f2(2.0f, 2.0f), f2(-2.0f, -2.0f));  // 2t, exact
  // coefficient i of Q (i = 8 .. 0) times 2^(-i - 1)
  float2 p = __ffma2_rn(w, f2(-0x1.321a48p-13f, -0x1.321a48p-13f), f2(0x1.068b28p-11f, 0x1.068b28p-11f));
  p = __ffma2_rn(w, p, f2(-0x1.0f9b0cp-10f, -0x1.0f9b0cp-10f));
  p = __ffma2_rn(w, p, f2(0x1.22bf86p-9f, 0x1.22bf86p-9f));
  p = __ffma2_rn(w, p, f2(-0x1.5424e0p-8f, -0x1.5424e0p-8f));
  p = __ffma2_rn(w, p, f2(0x1.999fc2p-7f, 0x1.999fc2p-7f));
  p = __ffma2_rn(w, p, f2(-0x1.000422p-5f, -0x1.000422p-5f));
  p = __ffma2_rn(w, p, f2(0x1.555558p-4f, 0x1.555558p-4f));
  p = __ffma2_rn(w, p, f2(-0x1.fffff8p-3f, -0x1.fffff8p-3f));
  const float2 lnf = __ffma2_rn(__fmul2_rn(w, w), p, w);
  return __ffma2_rn(ef, f2(0x1.62e4p+0f, 0x1.62e4p+0f),
                    __ffma2_rn(ef, f2(0x1.7f7d1cp-19f, 0x1.7f7d1cp-19f), lnf));
}

// The circle points of the angle words w0, w1 before the half turn of their
// bit 31 (the caller applies it as the sign of the radius): the position
// r = (bits 29..8) 2^-23 - 1/4 in [-1/4, 1/4) from the bits (0.5 + w 2^-23
// and its difference with 3/4 are exact), Taylor polynomials of sin(pi r)
// (to r^9) and cos(pi r) (to r^10) with coefficients (-1)^j pi^n/n! rounded
// to FP32, then (x, y) -> (-y, x) when bit 30 is set.
__device__ __forceinline__ void circle_x2(uint32_t w0, uint32_t w1, float2* x_out,
                                          float2* y_out) {
  const float2 h = f2(__uint_as_float(0x3F000000u | ((w0 >> 7) & 0x007FFFFEu)),
                      __uint_as_float(0x3F000000u | ((w1 >> 7) & 0x007FFFFEu)));
  const float2 r = __fadd2_rn(h, f2(-0.75f, -0.75f));
  const float2 r2 = __fmul2_rn(r, r);
  float2 sp = __ffma2_rn(r2, f2(0x1.507834p-4f, 0x1.507834p-4f), f2(-0x1.32d2ccp-1f, -0x1.32d2ccp-1f));
  sp = __ffma2_rn(r2, sp, f2(0x1.466bc6p+1f, 0x1.466bc6p+1f));
  sp = __ffma2_rn(r2, sp, f2(-0x1.4abbcep+2f, -0x1.4abbcep+2f));
  sp = __ffma2_rn(r2, sp, f2(0x1.921fb6p+1f, 0x1.921fb6p+1f));
  const float2 sn = __fmul2_rn(r, sp);
  float2 cp = __ffma2_rn(r2, f2(-0x1.a6d1f2p-6f, -0x1.a6d1f2p-6f), f2(0x1.e1f506p-3f, 0x1.e1f506p-3f));
  cp = __ffma2_rn(r2, cp, f2(-0x1.55d3c8p+0f, -0x1.55d3c8p+0f));
  cp = __ffma2_rn(r2, cp, f2(0x1.03c1f0p+2f, 0x1.03c1f0p+2f));
  cp = __ffma2_rn(r2, cp, f2(-0x1.3bd3ccp+2f, -0x1.3bd3ccp+2f));
  const float2 cs = __ffma2_rn(r2, cp, f2(1.0f, 1.0f));
  const bool q0 = (w0 & 0x40000000u) != 0u, q1 = (w1 & 0x40000000u) != 0u;
  *x_out = f2(q0 ? -sn.x : cs.x, q1 ? -sn.y : cs.y);
  *y_out = f2(q0 ? cs.x : sn.x, q1 ? cs.y : sn.y);
}

// Box-Muller of the word pairs (x.x, x.y) and (x.z, x.w), as (z0, z1, z2, z3):
// u1 = ((xa >> 8) + 1) 2^-24, rho = sqrt(-2 ln u1), (X, Y) the circle point
// of xb, (z_even, z_odd) = rho (X, Y).
__device__ __forceinline__ float4 box_muller_x2(uint4 x) {
  const float2 v = f2(__uint2float_rn((x.x >> 8) + 1u), __uint2float_rn((x.z >> 8) + 1u));  // exact
  const float2 nrho = neg_sqrt_neg_x2(ln2x_x2(v));
  // the half turn of bit 31 as the sign of the radius: (-rho) X = -(rho X)
  // exactly, signed zeros included
  const float2 rs = f2(__uint_as_float(__float_as_uint(nrho.x) ^ (~x.y & 0x80000000u)),
                       __uint_as_float(__float_as_uint(nrho.y) ^ (~x.w & 0x80000000u)));
  float2 cx, cy;
  circle_x2(x.y, x.w, &cx, &cy);
  const float2 zc = __fmul2_rn(rs, cx);
  const float2 zs = __fmul2_rn(rs, cy);
  return make_float4(zc.x, zs.x, zc.y, zs.y);
}

// The four uniform entries of one Philox call.
__device__ __forceinline__ float4 uniform_x4(uint4 x) {
  return make_float4(__fmul_rn(__uint2float_rn(x.x >> 8), 0x1p-24f),
                     __fmul_rn(__uint2float_rn(x.y >> 8), 0x1p-24f),
                     __fmul_rn(__uint2float_rn(x.z >> 8), 0x1p-24f),
                     __fmul_rn(__uint2float_rn(x.w >> 8), 0x1p-24f));
}

// The four Gaussian entries (r, 4j .. 4j+3).
template <class K>
__device__ __forceinline__ float4 gaussian4(const K& key, uint32_t r, uint32_t j) {
  return box_muller_x2(philox(j, r, key));
}

// The four uniform entries (r, 4j .. 4j+3).
template <class K>
__device__ __forceinline__ float4 uniform4(const K& key, uint32_t r, uint32_t j) {
  return uniform_x4(philox(j, r, key));
}

// The four Gaussian or uniform entries of row and column parts.
template <int DIST, class K>
__device__ __forceinline__ float4 entries4(const PhiloxRow& row, const PhiloxCol& col,
                                           const K& key) {
  const uint4 x = philox_join(row, col, key);
  return DIST == kUniform ? uniform_x4(x) : box_muller_x2(x);
}

// Sign bits of the 128 Rademacher entries (r, 128j .. 128j+127): bit b of
// word w belongs to column 128j + 32w + b; a set bit means -1.
template <class K>
__device__ __forceinline__ uint4 rademacher_bits(const K& key, uint32_t r, uint32_t j) {
  return philox(j, r, key);
}

// Four consecutive generated values (r, c0 .. c0+3), c0 % 4 == 0, as FP32
// (unquantized).
__device__ __forceinline__ float4 gen4(int dist, PhiloxKey key, uint32_t r, uint32_t c0) {
  if (dist == kRademacher) {
    const uint4 x = rademacher_bits(key, r, c0 >> 7);
    const uint32_t w = ((c0 >> 5) & 3u) == 0 ? x.x : ((c0 >> 5) & 3u) == 1 ? x.y
                     : ((c0 >> 5) & 3u) == 2 ? x.z : x.w;
    const uint32_t bits = w >> (c0 & 31u);
    return make_float4((bits & 1u) ? -1.f : 1.f, (bits & 2u) ? -1.f : 1.f,
                       (bits & 4u) ? -1.f : 1.f, (bits & 8u) ? -1.f : 1.f);
  }
  if (dist == kUniform) return uniform4(key, r, c0 >> 2);
  return gaussian4(key, r, c0 >> 2);
}

}  // namespace sk
