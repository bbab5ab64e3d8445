// What the two kernels of the integer tensor path share: how operands are tested, scaled and split, how the sums are joined.
#ifndef DETAG_DIGITS_CUH
#define DETAG_DIGITS_CUH

#include <cstdint>

#include "packed.cuh"
#include "pipeline.cuh"

namespace detag {

namespace {

// As bits of a coordinate's largest magnitude.  Mantissas from 1.988 on count as the next power of two, so that five balanced digits
// (at most 0x7F7F7F7F7F) hold every operand; maxima below 2^-90 leave the range of the float32 scale.
constexpr unsigned kRoundUp = 0x18000u, kSmallest = 0x12800000u;

// Digits of four workers' values x (+ rest, below 2^-18 of the coordinate's largest): digit k of all four in d[k].  The value z scale, at most 31 bits before
// the point, in two steps that float32 does exactly: its multiple of 2^14 next to it, and what is left in 1/256, each as the low bits
// of 1.5 * 2^23 plus it.  With the 40-bit integer q of both, q + 0x0080808080 has the balanced digits as bytes, all but the top one
// offset by 128.  No conversions: they run on a pipe a quarter as wide.
template <bool kRest>
__device__ __forceinline__ void digits_of(const F2 (&x)[2], const F2 (&rest)[2], float scale, uint32_t (&d)[5]) {
  uint32_t z[4], f[4];
#pragma unroll
  for (int v = 0; v < 4; v += 2) {
    const F2 high = fma2(x[v / 2], both(scale), both(206158430208.f));                          // 1.5 * 2^37
    F2 left = fma2(x[v / 2], both(scale), sub2(both(206158430208.f), high));
    if (kRest) left = fma2(rest[v / 2], both(scale), left);
    const F2 low = fma2(left, both(256.f), both(12583040.f));                                   // 1.5 * 2^23 + 128
    float h0, h1, f0, f1;
    unpack2(high, h0, h1);
    unpack2(low, f0, f1);
    f[v] = __float_as_uint(f0);
    f[v + 1] = __float_as_uint(f1);
    z[v] = (__float_as_uint(h0) << 14) + ((f[v] >> 8) + (0x00808080u - 0x4B4000u));
    z[v + 1] = (__float_as_uint(h1) << 14) + ((f[v + 1] >> 8) + (0x00808080u - 0x4B4000u));
  }
  const uint32_t ab = __byte_perm(z[0], z[1], 0x5140), cd = __byte_perm(z[2], z[3], 0x5140);
  const uint32_t ef = __byte_perm(z[0], z[1], 0x7362), gh = __byte_perm(z[2], z[3], 0x7362);
  d[0] = __byte_perm(__byte_perm(f[0], f[1], 0x0040), __byte_perm(f[2], f[3], 0x0040), 0x5410) ^ 0x80808080u;
  d[1] = __byte_perm(ab, cd, 0x5410) ^ 0x80808080u;
  d[2] = __byte_perm(ab, cd, 0x7632) ^ 0x80808080u;
  d[3] = __byte_perm(ef, gh, 0x5410) ^ 0x80808080u;
  d[4] = __byte_perm(ef, gh, 0x7632);
}

// Of four workers, `pitch` floats apart.
__device__ __forceinline__ void four_digits(const float* src, int pitch, float scale, uint32_t (&d)[5]) {
  const F2 x[2] = {pack2(src[0], src[pitch]), pack2(src[2 * pitch], src[3 * pitch])};
  digits_of<false>(x, x, scale, d);
}

// y + (g_new - g) (Algorithm 2's tracker update) as a float32 next to it: what the difference rounds off (Knuth's two-sum) is added again.  The
// sum may be far below its parts - all of it may be what was rounded off - but then y + fl(g_new - g) is exact (Sterbenz: the two are
// within a factor of two of one another), and the result is the sum rounded once; otherwise it is off by some ulps.
__device__ __forceinline__ float fold_value(float y, float g_new, float g) {
  const float t = g_new - g, tb = t - g_new;  // tb: the part of t that stands for -g
  return (y + t) + ((g_new - (t - tb)) - (g + tb));
}

// Digits of the sums y + (g_new - g) of four workers, the three arrays `array` floats apart: x = fl(y + fl(g_new - g)) and both roundings'
// errors e1, e2 (exact).  Where the parts cancel e1 + e2 is exact too (e2 = 0), and elsewhere below 2^-22 of x, so that x and their sum
// rounded once are the sum to 2^-46 of itself.  digits_of wants the latter below 2^-18 of the coordinate's largest: kCancels where
// that is not known, and then the two are normalised (x becomes the float32 next to the sum; |e1 + e2| <= |x|, or x = 0).
template <bool kCancels>
__device__ __forceinline__ void four_fold_digits(const float* src, int array, int pitch, float scale, uint32_t (&d)[5]) {
  F2 x[2], rest[2];
#pragma unroll
  for (int v = 0; v < 2; ++v) {
    const float* const at = src + 2 * v * pitch;
    const F2 y = pack2(at[0], at[pitch]), b = pack2(at[array], at[array + pitch]), a = pack2(at[2 * array], at[2 * array + pitch]);
    const F2 t = sub2(b, a), tb = sub2(t, b);
    const F2 e1 = sub2(sub2(b, sub2(t, tb)), add2(a, tb));
    x[v] = add2(y, t);
    const F2 xt = sub2(x[v], y);
    rest[v] = add2(e1, add2(sub2(y, sub2(x[v], xt)), sub2(t, xt)));
    if (kCancels) {
      const F2 s = add2(x[v], rest[v]);
      rest[v] = sub2(rest[v], sub2(s, x[v]));
      x[v] = s;
    }
  }
  digits_of<true>(x, rest, scale, d);
}

// Smallest of the largest magnitudes of groups first, first + step, ... of `size` inputs (2, or a multiple of 4), read as Four and Two.
template <typename Four, typename Two, typename Value, typename Index>
__device__ __forceinline__ float group_low(Value value, const Index* guard, int groups, int size, int first, int step) {
  float low = __uint_as_float(0x7f800000u);
  if (size == 2) {
#pragma unroll 4
    for (int q = first; q < groups; q += step) {
      const Two at = *reinterpret_cast<const Two*>(guard + 2 * q);
      low = fminf(low, max_abs3(value(at.x), value(at.y), 0.f));
    }
    return low;
  }
  for (int q = first; q < groups; q += step) {
    float m = 0.f;
#pragma unroll 2
    for (int i = 0; i < size; i += 4) {
      const Four at = *reinterpret_cast<const Four*>(guard + q * size + i);
      m = max_abs3(max_abs3(m, value(at.x), value(at.y)), value(at.z), value(at.w));
    }
    low = fminf(low, m);
  }
  return low;
}

// Integer sums of the five weights -> one float64, exact but for the rounding of the lowest: a 64-bit integer below 2^51, in units
// of 256^5, added to the bits of 1.5 * 2^52 with the coordinate's scale in its exponent field (`magic_hi`: the upper word; `magic`:
// that number), which is then subtracted.  `hi` = s8 * 256 + s7, `low` = s5 + s4 / 256, rounded.  Up to 128 workers (not kBig) the rest
// fits 32 bits (3 * 128 * 2^14 * 256 < 2^31).
template <bool kBig>
__device__ __forceinline__ double join_sums(int hi, int s6, int low, int magic_hi, double magic) {
  if (kBig) {
    const long long lo = static_cast<long long>(s6) * 256 + (low + (static_cast<long long>(magic_hi) << 32));
    return __longlong_as_double(static_cast<long long>(hi) * 65536 + lo) - magic;
  }
  const int lo = s6 * 256 + low;
  const unsigned long long upper = static_cast<uint32_t>(magic_hi + (lo >> 31));
  return __longlong_as_double(static_cast<long long>(hi) * 65536 + static_cast<long long>(upper << 32 | static_cast<uint32_t>(lo))) - magic;
}

}  // namespace

}  // namespace detag
#endif  // DETAG_DIGITS_CUH
