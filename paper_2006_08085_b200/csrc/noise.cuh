// Counter-based standard-normal noise of the stochastic gradient oracle.
//
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, "Parallel Random Numbers: As Easy as 1, 2, 3",
// SC'11) with key (seed low word, seed high word) and counter (j low word, j high word,
// i / 4, step) gives four words r0..r3 for the workers 4q..4q+3 (q = i / 4) at global
// coordinate j.  (r0, r1) and (r2, r3) each feed one Box-Muller transform:
//   u_rad = (2 (r_even >> 9) + 1) * 2^-24 in (0,1),  u_ang = (r_odd >> 9) * 2^-23 in [0,1)
//   rad = sqrt(-2 ln u_rad);  first = rad cos(2 pi u_ang);  second = rad sin(2 pi u_ang)
// Both uniforms are exactly representable in float32 and are built with bit operations, no
// integer-to-float conversion.  The logarithm is an own float32 routine (below); the square root uses the
// reciprocal-square-root unit and sine/cosine the special-function unit on an argument reduced
// exactly to [-pi, pi).  Resulting absolute error of a normal: about 1e-6 (1 + |xi|).
#ifndef DETAG_NOISE_CUH
#define DETAG_NOISE_CUH

#include <cstdint>

#include "packed.cuh"

namespace detag {

struct Philox4 {
  uint32_t r0, r1, r2, r3;
};

__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, uint32_t k0,
                                                 uint32_t k1) {
  constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u, kW0 = 0x9E3779B9u, kW1 = 0xBB67AE85u;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned long long p0 = static_cast<unsigned long long>(kM0) * c0;  // one wide multiply: hi and lo
    const unsigned long long p1 = static_cast<unsigned long long>(kM1) * c2;
    const uint32_t hi0 = static_cast<uint32_t>(p0 >> 32), lo0 = static_cast<uint32_t>(p0);
    const uint32_t hi1 = static_cast<uint32_t>(p1 >> 32), lo1 = static_cast<uint32_t>(p1);
    c0 = hi1 ^ c1 ^ (k0 + static_cast<uint32_t>(round) * kW0);
    c1 = lo1;
    c2 = hi0 ^ c3 ^ (k1 + static_cast<uint32_t>(round) * kW1);
    c3 = lo0;
  }
  return Philox4{c0, c1, c2, c3};
}

// The same with the twenty round keys (k0 + round * W0, k1 + round * W1 alternating) laid out by the host in the launch
// parameters: each is then a constant-bank operand of the exclusive-or that uses it instead of an addition of its own.
__device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3,
                                                 const uint32_t (&round_key)[20]) {
  constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u;
#pragma unroll
  for (int round = 0; round < 10; ++round) {
    const unsigned long long p0 = static_cast<unsigned long long>(kM0) * c0;
    const unsigned long long p1 = static_cast<unsigned long long>(kM1) * c2;
    c0 = static_cast<uint32_t>(p1 >> 32) ^ c1 ^ round_key[2 * round];
    c1 = static_cast<uint32_t>(p1);
    c2 = static_cast<uint32_t>(p0 >> 32) ^ c3 ^ round_key[2 * round + 1];
    c3 = static_cast<uint32_t>(p0);
  }
  return Philox4{c0, c1, c2, c3};
}

// 1 + (r >> 9) 2^-23: the exponent bits of 1.0 come in from above as the word is shifted, one instruction for both.
__device__ __forceinline__ float one_to_two(uint32_t r) { return __uint_as_float(__funnelshift_r(r, 0x7fu, 9)); }

// -2 ln(u) for u = (2k+1) 2^-24, k = r >> 9, of two words, as Cody and Waite ("Software Manual for the Elementary Functions",
// 1980) lay a logarithm out: u = m 2^e, ln u = e ln 2 + ln m with ln 2 in two parts.  Own choices:
//  - m in [2/3, 4/3).  Of the intervals [c, 2 c) this is the one with the smallest largest |m - 1|: 1 - c = 2 c - 1.  m and u
//    differ in their exponent fields alone, by e, so e is the exponent field of u's bits less the bits of c; m - 1 is exact.
//  - The parts of ln 2 are its nearest float32 and the float32 next to what is left.  A fused multiply-add does not round e times
//    either, so the upper part needs no room for e, and what both leave out is below 2^-53.
//  - ln(1 + f) = f + f^2 r(f), r a degree-7 Chebyshev fit of (ln(1+f) - f) / f^2 on |f| <= 1/3.
// Relative error over all 2^23 arguments: at most 9.9e-8, 2.9e-8 rms.  The factor -2 is in the argument F = -2 f and in the
// coefficients, scaled by powers of two: the bits are those of -2 times the logarithm.
__device__ __forceinline__ F2 neg2_ln_unit(uint32_t r0, uint32_t r1) {
  float u0, u1;
  unpack2(add2(pack2(one_to_two(r0), one_to_two(r1)), both(-0x1.fffffep-1f)), u0, u1);  // (2k+1) 2^-24, exact
  const int b0 = __float_as_int(u0), b1 = __float_as_int(u1);
  constexpr int kTwoThirds = 0x3f2aaaab, kExponent = static_cast<int>(0xff800000u);     // the float's bits; sign and exponent field
  const int e0 = (b0 - kTwoThirds) & kExponent, e1 = (b1 - kTwoThirds) & kExponent;     // here e 2^23
  const F2 F = fma2(pack2(__int_as_float(b0 - e0), __int_as_float(b1 - e1)), both(-2.0f), both(2.0f));  // -2 f, f = m - 1, exact
  // -r(-F/2) / 2
  F2 r7 = both(0.13756538927555084f * 0x1p-8f);
  r7 = fma2(r7, F, both(0.1504942923784256f * 0x1p-7f));
  r7 = fma2(r7, F, both(0.1405421793460846f * 0x1p-6f));
  r7 = fma2(r7, F, both(0.16481579840183258f * 0x1p-5f));
  r7 = fma2(r7, F, both(0.2000732272863388f * 0x1p-4f));
  r7 = fma2(r7, F, both(0.25004205107688904f * 0x1p-3f));
  r7 = fma2(r7, F, both(0.33333271741867065f * 0x1p-2f));
  r7 = fma2(r7, F, both(0.49999985098838806f * 0x1p-1f));
  F2 ln = fma2(mul2(F, F), r7, F);
  const F2 ef = pack2(__int2float_rn(e0), __int2float_rn(e1));                          // exact
  constexpr double kLn2 = 0.69314718055994530942;
  constexpr float kUpper = static_cast<float>(kLn2), kLower = static_cast<float>(kLn2 - static_cast<double>(kUpper));
  ln = fma2(ef, both(-kLower * 0x1p-22f), ln);
  return fma2(ef, both(-kUpper * 0x1p-22f), ln);
}

// Approximate reciprocal square root of a normal number (rsqrtf() tests for subnormal arguments first).
__device__ __forceinline__ float rsqrt_normal(float v) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
  return r;
}

// Both Box-Muller transforms of a Philox call: (first, third) and (second, fourth) normal.
__device__ __forceinline__ void box_muller(const Philox4& r, F2& even, F2& odd) {
  const F2 t = neg2_ln_unit(r.r0, r.r2);  // 1.2e-7 .. 33.3
  float t0, t1, a0, a1;
  unpack2(t, t0, t1);
  const F2 rad = mul2(t, pack2(-rsqrt_normal(t0), -rsqrt_normal(t1)));                                              // negated
  const F2 theta = mul2(add2(pack2(one_to_two(r.r1), one_to_two(r.r3)), both(-1.5f)), both(6.283185307179586f));    // 2 pi u_ang - pi
  unpack2(theta, a0, a1);
  even = mul2(rad, pack2(__cosf(a0), __cosf(a1)));  // cos(2 pi u) = -cos(2 pi u - pi)
  odd = mul2(rad, pack2(__sinf(a0), __sinf(a1)));
}

// Standard normals of workers 4q..4q+3 at global coordinate j and noise step t.
__device__ __forceinline__ void normal_quad(const uint32_t (&round_key)[20], unsigned long long j, uint32_t q, uint32_t t, float (&xi)[4]) {
  F2 even, odd;
  box_muller(philox4x32_10(static_cast<uint32_t>(j), static_cast<uint32_t>(j >> 32), q, t, round_key), even, odd);
  unpack2(even, xi[0], xi[2]);
  unpack2(odd, xi[1], xi[3]);
}

// `scale` times those.
__device__ __forceinline__ void normal_quad(const uint32_t (&round_key)[20], unsigned long long j, uint32_t q, uint32_t t, float scale,
                                            float (&xi)[4]) {
  F2 even, odd;
  box_muller(philox4x32_10(static_cast<uint32_t>(j), static_cast<uint32_t>(j >> 32), q, t, round_key), even, odd);
  unpack2(mul2(even, both(scale)), xi[0], xi[2]);
  unpack2(mul2(odd, both(scale)), xi[1], xi[3]);
}

// `scale` times the normals of workers 4q..4q+7 at one coordinate.  The two calls differ in the third counter word alone: of
// the first round's products one is common and the other grows by the multiplier, of the second round's one is common.
__device__ __forceinline__ void normal_eight(const uint32_t (&round_key)[20], unsigned long long j, uint32_t q, uint32_t t, float scale,
                                             float (&xi)[8]) {
  constexpr uint32_t kM0 = 0xD2511F53u, kM1 = 0xCD9E8D57u;
  const unsigned long long pj = static_cast<unsigned long long>(kM0) * static_cast<uint32_t>(j);
  const uint32_t c2 = static_cast<uint32_t>(pj >> 32) ^ t ^ round_key[1], c3 = static_cast<uint32_t>(pj);
  const unsigned long long p1 = static_cast<unsigned long long>(kM1) * c2;
  unsigned long long pq = static_cast<unsigned long long>(kM1) * q;
#pragma unroll
  for (int h = 0; h < 2; ++h, pq += kM1) {
    const uint32_t c0 = static_cast<uint32_t>(pq >> 32) ^ static_cast<uint32_t>(j >> 32) ^ round_key[0];
    const unsigned long long p0 = static_cast<unsigned long long>(kM0) * c0;
    Philox4 r{static_cast<uint32_t>(p1 >> 32) ^ static_cast<uint32_t>(pq) ^ round_key[2], static_cast<uint32_t>(p1),
              static_cast<uint32_t>(p0 >> 32) ^ c3 ^ round_key[3], static_cast<uint32_t>(p0)};
#pragma unroll
    for (int round = 2; round < 10; ++round) {
      const unsigned long long a = static_cast<unsigned long long>(kM0) * r.r0;
      const unsigned long long b = static_cast<unsigned long long>(kM1) * r.r2;
      r.r0 = static_cast<uint32_t>(b >> 32) ^ r.r1 ^ round_key[2 * round];
      r.r1 = static_cast<uint32_t>(b);
      r.r2 = static_cast<uint32_t>(a >> 32) ^ r.r3 ^ round_key[2 * round + 1];
      r.r3 = static_cast<uint32_t>(a);
    }
    F2 even, odd;
    box_muller(r, even, odd);
    unpack2(mul2(even, both(scale)), xi[4 * h], xi[4 * h + 2]);
    unpack2(mul2(odd, both(scale)), xi[4 * h + 1], xi[4 * h + 3]);
  }
}

}  // namespace detag
#endif  // DETAG_NOISE_CUH
