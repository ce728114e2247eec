// fixpoint.h - block fixed point for the FP64 half Dslash: digits, exponents and products.
//
// GB300 runs 2 FP64 multiply-adds per clock and SM, so the 288 of one output site cost 144 clocks, six
// times what the site's 1248 bytes need from HBM.  Its 32 x 32 + 64-bit integer multiply-add runs 64 lanes
// per clock and is exact.  A link entry and a vector component therefore enter the products as fixed-point
// numbers F = H 2^28 + L (H and L of one sign, |L| < 2^28):
//   - links in units of 2^-57 (|1/2 eta bc U| <= 1/2, |H| <= 2^28 (1 + 2^-8)), digitised when the gauge field
//     is set;
//   - vectors against the largest component among the site's eight neighbours (|H| < 2^30), digitised when
//     they are read.
// One complex product takes 12 integer multiply-adds (the H H products exactly, the H L products exactly in
// an accumulator of their own, L L dropped), 864 per site: 13.5 clocks, beside about 20 shifts and logic
// operations per component for the digits.  With one exponent per output site all products add up as
// integers, so the sum does not depend on its order, and one conversion per component rounds it to FP64.
//
// Accuracy.  With 2^E the power of two at or below the largest neighbouring component and m_mu 2^E the largest one of
// direction mu's two neighbours, the steps before that rounding err per real component by at most 2^(E-58) times
// 12 sum_mu m_mu (links rounded to 2^-58), 20 (vectors truncated at 2^(E-57) against rows of norm 1/2), 48 (48 dropped
// L L products) and 2 (the H L sums rounded once per direction).  What counts for the result is S, the sum of
// the magnitudes of the component's own 48 products, which may be far smaller: links that do not mix the
// colours beside colours of different size, or entries below 2^-57 of their unit.  The digits are used where that
// error is below 21 x 2^-53 S, that of the 25 roundings of an FP64 multiply-add chain; S is bounded from below by the
// eight hops' magnitudes (fix_hop_words, fix_needed).  A component short of it is computed in FP64: on rough fields with
// Gaussian vectors (S of 5 to 10 2^E, 0.1 to 0.26 2^E needed) one in about 2 million.  Against quad precision the
// hop's error is 4.9e-17, that of the FP64 multiply-adds 1.7e-16 (Gaussian vectors, 8 x 6 x 4 x 6).
//
// The integers' ranges.  A row or column of 1/2 U has norm 1/2; the format takes up to kFixMaxNorm = 0.501, so
// that by the Cauchy-Schwarz inequality every partial sum of a component's 48 products is at most
// 8 x 0.501 x sqrt(6) = 9.82 times 2^29 2^30 in units of H H: 2^62.3.  The 24 H L products of one thread's two
// hops are at most 12 2^28 (2^30 + 2^28.1) < 2^62.
//
// What else does not fit (a link with a row or column of larger norm or not finite, neighbours whose largest
// component lies outside 2^-800 .. 2^800 or is not finite) marks the site, which is then computed in FP64.
//
// Plain integer arithmetic: the host build, used by the tests, gives the device's bits.
#pragma once

#include <stdint.h>
#include <string.h>

#if defined(__CUDACC__)
#define LQCD_FIX_HD __host__ __device__ __forceinline__
#else
#define LQCD_FIX_HD inline
#endif

namespace lqcd {

constexpr int kFixLow = 28;  // bits of the low digit
constexpr int kFixMinE = 1023 - 800, kFixMaxE = 1023 + 800;
constexpr double kFixMaxNorm = 0.501;

struct Fix2 {
  int h, l;
};

// Exponents: a component with biased exponent e is M 2^(e - 1023 - 63), M its mantissa as a 64-bit word with
// the top bit set.  Against the block exponent E its digits are F = M >> (6 + E - e), value F 2^(E - 1023 - 57).  A
// link entry is F 2^-57.  The sums are in units of H H, 2^56 F F: value = sum 2^(E - kFixUnit).
constexpr int kFixUnit = 1023 + 57 + 57 - 2 * kFixLow;

LQCD_FIX_HD int fix_hi(double x) {
#if defined(__CUDA_ARCH__)
  return __double2hiint(x);
#else
  int64_t b;
  memcpy(&b, &x, 8);
  return (int)(b >> 32);
#endif
}
LQCD_FIX_HD uint32_t fix_lo(double x) {
#if defined(__CUDA_ARCH__)
  return (uint32_t)__double2loint(x);
#else
  uint64_t b;
  memcpy(&b, &x, 8);
  return (uint32_t)b;
#endif
}
LQCD_FIX_HD uint32_t fix_shr32(uint32_t a, int n) {  // n >= 0; 0 from n = 32 on
#if defined(__CUDA_ARCH__)
  uint32_t r;
  asm("shr.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(n));
  return r;
#else
  return n < 32 ? a >> n : 0u;
#endif
}
LQCD_FIX_HD uint64_t fix_shr64(uint64_t a, int n) {  // n >= 0; 0 from n = 64 on
#if defined(__CUDA_ARCH__)
  uint64_t r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(a), "r"(n));
  return r;
#else
  return n < 64 ? a >> n : 0u;
#endif
}
LQCD_FIX_HD uint32_t fix_low_word(uint32_t lo, uint32_t hi, int n) {  // of (hi : lo) >> min(n, 32), n >= 0
#if defined(__CUDA_ARCH__)
  return __funnelshift_rc(lo, hi, n);
#else
  return (uint32_t)((((uint64_t)hi << 32) | lo) >> (n < 32 ? n : 32));
#endif
}

// the upper half of the mantissa word M (the lower half is lo << 11)
LQCD_FIX_HD uint32_t fix_mantissa_hi(int hi, uint32_t lo) { return ((uint32_t)hi << 11 | lo >> 21) | 0x80000000u; }
LQCD_FIX_HD int fix_exponent(int hi) { return (int)(((uint32_t)hi << 1) >> 21); }

// One component against block exponent E, its own exponent or larger; FLIP negates it.  e = 0 (zero) gives
// 0: E >= kFixMinE.
template <bool FLIP>
LQCD_FIX_HD Fix2 fix_component(double x, int E) {
  const int hi = fix_hi(x);
  const uint32_t lo = fix_lo(x);
  const int n = E + 6 - fix_exponent(hi);  // F = (mh : ml) >> n, n >= 6
  const uint32_t mh = fix_mantissa_hi(hi, lo), ml = lo << 11;
  const uint32_t h = fix_shr32(mh, n - 4);
  const uint32_t l = fix_shr32(fix_low_word(ml, mh, n), n > 32 ? n - 32 : 0) & ((1u << kFixLow) - 1);
  const int sg = ((FLIP ? ~hi : hi) >> 31) | 1;
  return Fix2{(int)h * sg, (int)l * sg};
}

// A link entry's digits, rounded; |u| <= kFixMaxNorm
LQCD_FIX_HD Fix2 fix_link_entry(double u) {
  const int hi = fix_hi(u), s = hi >> 31;
  const uint32_t lo = fix_lo(u);
  const uint64_t M = (uint64_t)fix_mantissa_hi(hi, lo) << 32 | lo << 11;
  const uint64_t F = (fix_shr64(M, 5 + 1023 - fix_exponent(hi)) + 1) >> 1;
  return Fix2{((int)(F >> kFixLow) ^ s) - s, (((int)F & ((1 << kFixLow) - 1)) ^ s) - s};
}

// Every row and column of the (folded) link within the format; false for NaN and infinities.  u[j]: entry j
// of the row-major matrix, with members x, y (real and imaginary part), in FP64 or rounded to FP32 (the limit then moves by
// 10^-6 of itself, far from what the integers hold): in FP64 the check of 32^3x8's links makes
// lqcd_set_gauge 50 us longer (550 instead of 500) on GB300's FP64 pipe.
template <typename C>
LQCD_FIX_HD bool fix_link_fits(const C (&u)[9]) {
  typedef decltype(u[0].x + u[0].x) T;
  bool ok = true;
  for (int a = 0; a < 3; ++a) {
    T r = 0, c = 0;
    for (int b = 0; b < 3; ++b) {
      r += u[3 * a + b].x * u[3 * a + b].x + u[3 * a + b].y * u[3 * a + b].y;
      c += u[3 * b + a].x * u[3 * b + a].x + u[3 * b + a].y * u[3 * b + a].y;
    }
    ok = ok && r <= (T)(kFixMaxNorm * kFixMaxNorm) && c <= (T)(kFixMaxNorm * kFixMaxNorm);
  }
  return ok;
}

// What the block exponent is taken from: the largest high word of n components' magnitudes, or -1 where the
// largest one is not zero but too small for the format.
template <int N>
LQCD_FIX_HD int fix_max_word(const double (&v)[N]) {
  int m = 0;
  for (int c = 0; c < N; ++c) {
    const int w = fix_hi(v[c]) & 0x7fffffff;
    m = w > m ? w : m;
  }
  if (m < (kFixMinE << 20)) {
    uint32_t any = (uint32_t)m;
    for (int c = 0; c < N; ++c) any |= fix_lo(v[c]);
    m = any ? -1 : 0;
  }
  return m;
}

// The block exponent from the max words of a site's neighbours; -1 outside the format.
template <int N>
LQCD_FIX_HD int fix_block_exponent(const int (&w)[N]) {
  int m = 0, any = 0;
  for (int q = 0; q < N; ++q) {
    m = w[q] > m ? w[q] : m;
    any |= w[q];
  }
  const int E = m >> 20;
  return any < 0 || E > kFixMaxE ? -1 : (E < kFixMinE ? kFixMinE : E);
}

// The least sum over the eight hops of the magnitudes of their sums' upper 32 bits (fix_hop_words) with which a
// component's digits are accurate enough: (70 + 12 sum_mu m_mu) 2^-58 <= 21 x 2^-53 S / 2^E, S / 2^E = words 2^-26, so
// words >= (70 + 12 sum m) 2^26 / 672; here 2^20 (7 + 1.25 sum m), more than 4 % above it, which takes what the
// upper words leave out.  w: the max words of the four directions.
LQCD_FIX_HD uint32_t fix_needed(const int (&w)[4], int E) {
  uint32_t m = 0;
  for (int q = 0; q < 4; ++q) m += fix_shr32(1u << 20 | ((uint32_t)w[q] & 0xfffffu), E - (w[q] >> 20));
  return (7u << 20) + m + (m >> 2);
}
LQCD_FIX_HD int fix_upper(int64_t sum) { return (int)(sum >> 32); }
// |a hop's sum| is at most its products' magnitudes together.  fwd, both: upper words after the forward hop and both
LQCD_FIX_HD uint32_t fix_hop_words(int fwd, int both) {
  const uint32_t f = (uint32_t)fwd, b = (uint32_t)both - f;
  return (fwd < 0 ? 0u - f : f) + ((int)b < 0 ? 0u - b : b);
}

// hh += the H H product, x += the two H L products of (ah, al) and b
LQCD_FIX_HD void fix_mac(int64_t& hh, int64_t& x, int ah, int al, Fix2 b) {
#if defined(__CUDA_ARCH__)
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(hh) : "r"(ah), "r"(b.h));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(x) : "r"(ah), "r"(b.l));
  asm("mad.wide.s32 %0, %1, %2, %0;" : "+l"(x) : "r"(al), "r"(b.h));
#else
  hh += (int64_t)ah * b.h;
  x += (int64_t)ah * b.l;
  x += (int64_t)al * b.h;
#endif
}

}  // namespace lqcd
