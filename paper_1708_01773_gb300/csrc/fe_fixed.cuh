// Fixed-point arithmetic for the FP64 forms of the contractions.
//
// GB300 issues FP64 at 2 lanes per clock per SM but 32 x 32 + 64 bit integer
// multiply-adds at 32 or more. A sum of K products of operands that are known
// to be bounded is therefore formed exactly in integers: each operand is a
// signed B-bit integer v = hi 2^L + lo (lo in [-2^(L-1), 2^(L-1))), a product
// takes three wide multiply-adds (hi hi, hi lo + lo hi; lo lo is left out
// with L = 30 but where it can be a square, or summed in FP32 with L = 32), and the sums need no rounding
// until they are converted to a double once.
// Bounds: the hi hi sums of K products stay below K 2^(2B - 2L) < 2^63; the
// cross sums are drained into them after at most S products, S 2^B < 2^63.
// L = 30, B = 59: K <= 30, S <= 12 (Q1; Q2 elasticity). L = 32, B = 59:
// K <= 486, S <= 12 (longer sums: without lo lo their error, sqrt(K)/12 units
// of 2^(2L), would exceed the rounding of the operands).
#pragma once

#include <cstdint>

namespace feasm {

constexpr int kFixBits = 59;       // B
constexpr int kFixDrainEvery = 12; // S

// d += a * b, 32 x 32 -> 64 bit signed
__device__ __forceinline__ void mad_wide(int64_t& d, int a, int b) {
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(d) : "r"(a), "r"(b));
}

// hi/lo limbs of v, |v| <= 2^60
template <int L>
__device__ __forceinline__ int2 fix_limbs(int64_t v) {
  if (L == 32) {
    const int l = int(uint32_t(uint64_t(v)));
    return make_int2(int(v >> 32) - (l >> 31), l);
  }
  const int h = int((v + (1 << 29)) >> 30);
  return make_int2(h, int(uint32_t(uint64_t(v))) - int(uint32_t(h) << 30));
}

// x 2^scale rounded to an integer, for |x| 2^scale < 2^62; x finite. Values
// below half a unit (denormals among them) give 0.
__device__ __forceinline__ int64_t fix_quantise(double x, int scale) {
  const uint64_t u = uint64_t(__double_as_longlong(x));
  const int e = int((u >> 52) & 0x7ffu);
  const uint64_t m = (u & 0xfffffffffffffull) | (1ull << 52);
  const int sh = e - 1075 + scale;
  uint64_t a;
  if (sh >= 0) {
    a = m << (sh & 63);
  } else {
    a = sh > -55 ? ((m >> (-sh - 1)) + 1) >> 1 : 0ull;
  }
  if (e == 0) a = 0;
  return (u >> 63) ? -int64_t(a) : int64_t(a);
}

// The two accumulators of a sum of products; value = hh 2^(2L) + x 2^L in units
// of the operands' product.
template <int L>
struct FixAcc {
  int64_t hh, x;
  __device__ __forceinline__ void zero() {
    hh = 0;
    x = 0;
  }
  __device__ __forceinline__ void add(int2 a, int2 b) {
    mad_wide(hh, a.x, b.x);
    mad_wide(x, a.x, b.y);
    mad_wide(x, a.y, b.x);
  }
  __device__ __forceinline__ void drain() {
    hh += x >> L;
    x &= (int64_t(1) << L) - 1;
  }
  // value / 2^(2L + sh), 1 <= sh <= 62, rounded to nearest from the sum's full
  // length. (Rounded to 2L first, half of all values are ties where one more bit
  // goes; rounding those up moves every operand the same way, by a quarter unit on
  // average, and leaves a residual of translations in every cell.)
  __device__ __forceinline__ int64_t get_shifted(int sh) const { return (((hh + (x >> L)) >> (sh - 1)) + 1) >> 1; }
  // After drain(): adds an exact sum of lo lo products
  __device__ __forceinline__ void add_low(int64_t lolo) {
    x += (lolo + (int64_t(1) << (L - 1))) >> L;
    drain();
  }
  // After drain(): adds a sum of lo lo products, |lolo| < 2^92
  __device__ __forceinline__ void add_low(float lolo) {
    x += __float2ll_rn(lolo * (L == 32 ? 0x1p-32f : 0x1p-30f));
    drain();
  }
  // After drain(): the leading sign bits of the value that are free to shift out.
  __device__ __forceinline__ uint32_t magnitude() const {
    const int h = int(hh >> 32);
    return uint32_t(h ^ (h >> 31));
  }
  // After drain(): value 2^(g - 2 - 2L), 0 <= g <= 31, rounded (not cut off:
  // a bias of the same sign in every entry of a matrix, however small, moves
  // its softest modes): the 64 + L bits of (hh, x) shifted left by g - 2.
  __device__ __forceinline__ int64_t get(int g) const {
    const uint32_t w2 = uint32_t(uint64_t(hh) >> 32), w1 = uint32_t(uint64_t(hh));
    const uint32_t v2 = uint32_t(int(w2) >> 2), v1 = __funnelshift_r(w1, w2, 2);
    const uint32_t v0 = (w1 << 30) | (uint32_t(uint64_t(x)) >> (L - 30));
    return int64_t((uint64_t(__funnelshift_l(v1, v2, g)) << 32) | __funnelshift_l(v0, v1, g)) + int64_t((v0 << g) >> 31);
  }
};

// Shift g for get(g) that brings values of the given magnitude() (the bitwise
// or over the values that share the shift) below 2^61.
__device__ __forceinline__ int fix_shift(uint32_t magnitude) { return min(__clz(int(magnitude)) - 1, 31); }

// v = h 2^32 + l with signed halves, |v| < 2^63 - 2^31
__device__ __forceinline__ void fix_halves(int64_t v, int& h, int& l) {
  l = int(uint32_t(uint64_t(v)));
  h = int(v >> 32) - (l >> 31);
}

// a m / 2^64 (m = mh 2^32 + ml with signed halves, |m| <= 2^61, |a| < 2^63), to about one unit
__device__ __forceinline__ int64_t fix_mul(int64_t a, int mh, int ml) {
  int ah, al;
  fix_halves(a, ah, al);
  int64_t c = int64_t(1) << 31, h = 0;
  mad_wide(c, ah, ml);
  mad_wide(c, al, mh);
  mad_wide(h, ah, mh);
  return h + int(c >> 32);
}

// t-th pair (a, b), a <= b, b-major: t = b (b + 1) / 2 + a, t < 2^20
__device__ __forceinline__ void fix_pair(int t, int& a, int& b) {
  b = int((sqrtf(float(8 * t + 1)) - 1.f) * 0.5f);
  if (b * (b + 1) / 2 > t) --b;
  if ((b + 1) * (b + 2) / 2 <= t) ++b;
  a = t - b * (b + 1) / 2;
}

// 1 / sqrt(x) = y 2^-k2 for a positive normal x: the FP32 reciprocal square
// root of x's mantissa (relative error h0 < 2^-21) and one step of
// y (1 + h/2 + 3/8 h^2), h = 1 - x y^2, which leaves 5/16 h^3 < 2^-61; `odd`
// is set for any other x.
__device__ __forceinline__ double fix_rsqrt(double x, int& k2, bool& odd) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int eb = hi >> 20;                  // sign and exponent
  odd |= eb < 1 || eb > 2046;
  const int e = (eb & 0x7ff) - 1023;
  k2 = e >> 1;
  const int r = e & 1;                      // mantissa times 2^r in [1, 4)
  const double m = __hiloint2double((hi & 0xfffff) | ((1023 + r) << 20), lo);
  const float mf = __uint_as_float(uint32_t((127 + r) << 23) | (uint32_t(hi & 0xfffff) << 3) | (uint32_t(lo) >> 29));
  const uint32_t yu = __float_as_uint(rsqrtf(mf));  // in (0.5, 1]
  const double y = __hiloint2double(int((yu >> 3) + 0x38000000u), int(yu << 29));
  const double h = fma(-m, y * y, 1.0);
  return fma(y * h, fma(0.375, h, 0.5), y);
}

static __device__ __noinline__ double reciprocal_slow(double x) { return 1.0 / x; }
// 1 / x: the FP32 reciprocal of the mantissa and r (1 + h + h^2), h = 1 - m r, which leaves h^3 < 2^-60
__device__ __forceinline__ double reciprocal(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x), eb = (hi >> 20) & 0x7ff;
  if (eb < 2 || eb > 2044) return reciprocal_slow(x);
  const double m = __hiloint2double((hi & 0x800fffff) | (1023 << 20), lo);
  const float mf = __uint_as_float((uint32_t(hi) & 0x80000000u) | (127u << 23) | (uint32_t(hi & 0xfffff) << 3) | (uint32_t(lo) >> 29));
  const uint32_t ru = __float_as_uint(__frcp_rn(mf));
  const double r = __hiloint2double(int((ru & 0x80000000u) | (((ru & 0x7fffffffu) >> 3) + 0x38000000u)), int(ru << 29));
  const double h = fma(-m, r, 1.0);
  const double y = fma(r, fma(h, h, h), r);
  return __hiloint2double(__double2hiint(y) - ((eb - 1023) << 20), __double2loint(y));
}

// x 2^k by exponent arithmetic, for |x| in [1/2, 1] and |k| < 1000
__device__ __forceinline__ double fix_scale2(double x, int k) {
  return __hiloint2double(__double2hiint(x) + int(uint32_t(k) << 20), __double2loint(x));
}

// I 2^ex as a double (nearest, ties away from zero), |I| < 2^63, for results
// within the normal range (ex in [-960, 900]; the caller checks). In two steps:
// the part of the exponent field that does not depend on I, then the
// conversion; |I| < 2^32 (zero among them) takes the general path.
__device__ __forceinline__ int fix_exponent(int ex) { return (ex + 62 + 1022) << 20; }
static __device__ __noinline__ double fix_to_double_small(int64_t I, int field) {
  if (I == 0) return 0.0;
  const uint64_t s = uint64_t(I >> 63);
  const uint64_t mag = (uint64_t(I) ^ s) - s;
  const int sh = __clzll(static_cast<long long>(mag)) - 1;
  const uint64_t n = (mag << sh) + 0x200u;
  return __longlong_as_double(static_cast<long long>(((n >> 10) + (uint64_t(uint32_t(field - (sh << 20))) << 32)) |
                                                     (s & 0x8000000000000000ull)));
}
__device__ __forceinline__ double fix_to_double(int64_t I, int field) {
  const int s = int(I >> 63);
  const uint64_t mag = (uint64_t(I) ^ uint64_t(int64_t(s))) - uint64_t(int64_t(s));
  const uint32_t hi = uint32_t(mag >> 32), lo = uint32_t(mag);
  if (hi == 0) return fix_to_double_small(I, field);
  const int sh = __clz(int(hi)) - 1;  // leading one to bit 62
  const uint64_t n = ((uint64_t(__funnelshift_l(lo, hi, sh)) << 32) | (lo << sh)) + 0x200u;
  const uint32_t nh = uint32_t(n >> 32), nl = uint32_t(n);
  // n >> 10 has its leading one at bit 52, which adds 1 to the exponent field
  const int top = int(nh >> 10) + (sh * -(1 << 20) + field);
  return __hiloint2double(top | (s & int(0x80000000u)), int(__funnelshift_r(nl, nh, 10)));
}

}  // namespace feasm
