// kp_arith.cuh -- rules of the loop kernel that give a costlier form's answer by
// other arithmetic: the division of a sample key by lambda, the acceptance
// thresholds and draws without a division, the clearance test in integers.
// Compiled for the device and, for their tests, for the host.
#pragma once

#include <cfenv>
#include <cmath>
#include <cstdint>
#include <cstring>

namespace kp {

#define KP_HD __host__ __device__ __forceinline__

// Explicitly rounded operations and bit patterns on either side (the host's are
// compiled without contraction of products into sums).
namespace hd {
#ifdef __CUDA_ARCH__
KP_HD float mul(float a, float b) { return __fmul_rn(a, b); }
KP_HD float add(float a, float b) { return __fadd_rn(a, b); }
KP_HD float fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
KP_HD float fma_up(float a, float b, float c) { return __fmaf_ru(a, b, c); }
KP_HD double add(double a, double b) { return __dadd_rn(a, b); }
KP_HD double div(double a, double b) { return __ddiv_rn(a, b); }
KP_HD double fma(double a, double b, double c) { return __fma_rn(a, b, c); }
KP_HD int bits(float v) { return __float_as_int(v); }
KP_HD float f32(int v) { return __int_as_float(v); }
KP_HD long long bits(double v) { return __double_as_longlong(v); }
KP_HD double f64(long long v) { return __longlong_as_double(v); }
KP_HD uint32_t mul_high(uint32_t a, uint32_t b) { return __umulhi(a, b); }
KP_HD int top_bit(uint32_t v) { return 31 - __clz((int)v); }
#else
template <class To, class From>
KP_HD To same_bits(From v) {
  To r;
  std::memcpy(&r, &v, sizeof r);
  return r;
}
KP_HD float mul(float a, float b) { return a * b; }
KP_HD float add(float a, float b) { return a + b; }
KP_HD float fma(float a, float b, float c) { return std::fmaf(a, b, c); }
KP_HD float fma_up(float a, float b, float c) {
  const int mode = std::fegetround();
  std::fesetround(FE_UPWARD);
  volatile float r = std::fmaf(a, b, c);
  std::fesetround(mode);
  return r;
}
KP_HD double add(double a, double b) { return a + b; }
KP_HD double div(double a, double b) { return a / b; }
KP_HD double fma(double a, double b, double c) { return std::fma(a, b, c); }
KP_HD int bits(float v) { return same_bits<int>(v); }
KP_HD float f32(int v) { return same_bits<float>(v); }
KP_HD long long bits(double v) { return same_bits<long long>(v); }
KP_HD double f64(long long v) { return same_bits<double>(v); }
KP_HD uint32_t mul_high(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
KP_HD int top_bit(uint32_t v) {
  int n = 0;
  while (v >>= 1) ++n;
  return n;
}
#endif
KP_HD int high(double v) { return (int)(bits(v) >> 32); }
}  // namespace hd

// Division of a sample key by the pass's lambda (at most 1024) by a
// multiplication: for lam in [2^s, 2^(s+1)) and mul = ceil(2^(31+s) / lam), key
// / lam = (key mul) >> (31 + s) for every key below 2^30 (the product exceeds
// the quotient's by key (mul lam - 2^(31+s)) / lam < key, less than the 2^(31+s)
// / lam that is left).  Two 32-bit divisions a pass and thread instead of one a
// sample: mul's quotient in two steps, 2^31 = a lam + b, 2^s b = c lam + d.
struct KeyDiv {
  int lam, shift;
  uint32_t mul;
  KP_HD explicit KeyDiv(int l) : lam(l), shift(0), mul(0) {
    if (l > 0) {
      const uint32_t u = (uint32_t)l;
      shift = hd::top_bit(u);
      const uint32_t a = 0x80000000u / u, b = 0x80000000u - a * u;
      const uint32_t c = (b << shift) / u, d = (b << shift) - c * u;
      mul = (a << shift) + c + (d != 0u ? 1u : 0u);
    }
  }
  KP_HD int quot(int key) const { return (int)(hd::mul_high((uint32_t)key << 1, mul) >> shift); }
};

// Whether a distance d (cells) is at most 1 + q / 16, q a clearance byte (0:
// none): 16 d - 16 rounded up to an integer, in the low bits of 2^23 + it,
// against q.
KP_HD bool within_clearance(float d, int q) {
  const int e = hd::bits(hd::fma_up(d, 16.0f, 8388592.0f));
  return q != 0 && e - 0x4B000000 <= q;
}

// The score that stands for none (outside R_avail), told from all others by its
// high word: a score is not negative, but one that is not a number (an infinite
// delta) has the sign bit set.
constexpr double KP_NO_SCORE = -1.0;
KP_HD bool no_score(int score_hi) { return score_hi == (int)0xbff00000; }

// floor(min(p, 1) 2^32) of a positive p, from its bits: the mantissa shifted
// down by as much as its last place lies below 2^-32 (an FP64 instruction
// takes 64 clocks here, and this was four of them).
KP_HD uint64_t threshold_of(double p) {
  const uint64_t bits = (uint64_t)hd::bits(p);
  const int e = (int)(bits >> 52) - 1023;  // p in [2^e, 2^(e+1))
  if (e >= 0) return 1ull << 32;           // infinities too
  const uint64_t mant = (bits & 0xfffffffffffffull) | (1ull << 52);
  const int down = 20 - e;                 // 52 - 32 - e
  return down < 64 ? mant >> down : 0ull;
}

// The sum of Eq. 5 and what the thresholds and draws take from it.
struct ScoreSum {
  double sum, inv;    // inv: 1 / sum, 0 where the division is always taken
  float inv_m, eps32; // inv's mantissa; eps
  int inv_e;          // inv's exponent (without an inverse: so large that a draw
                      // takes the threshold itself)
};

// inv only for a sum that is a number between 2^-900 and 2^900.
KP_HD ScoreSum score_sum_of(double sum, double eps) {
  ScoreSum s;
  const int e = (hd::high(sum) >> 20) - 1023;  // of a positive number
  s.sum = sum;
  const double inv = e >= -900 && e <= 900 ? hd::div(1.0, sum) : 0.0;
  s.inv = inv;
  s.inv_e = inv > 0.0 ? (hd::high(inv) >> 20) - 1023 : 1 << 16;
  s.inv_m = inv > 0.0 ? (float)hd::f64((hd::bits(inv) & 0xfffffffffffffll) | 0x3ff0000000000000ll) : 1.0f;
  s.eps32 = (float)eps;
  return s;
}

// The acceptance threshold of a region with this score (none: outside R_avail,
// P_accept = 1): threshold_of(score / sum + eps), eps below 1, or
// threshold_of(eps) when the sum is not positive.  inv = 1 / sum gives it without
// the division (573 clocks and about ten FP64 operations, of which an SM does
// two a clock): score inv + eps in one rounding is within 4 units in the last
// place of the value it stands for (half from inv, half each from the two
// roundings there and one here, at most doubled by a binade), so where 16 units
// more or less make no difference to the threshold it is the same one.
KP_HD uint64_t accept_threshold(double score, double sum, double inv, double eps) {
  if (no_score(hd::high(score))) return 1ull << 32;
  if (hd::high(inv) != 0) {
    const long long near = hd::bits(hd::fma(score, inv, eps));
    const uint64_t lo = threshold_of(hd::f64(near - 16));
    if (lo == threshold_of(hd::f64(near + 16))) return lo;
  }
  return threshold_of(sum > 0.0 ? hd::add(hd::div(score, sum), eps) : eps);
}

// Whether the draw w of a node is below its region's accept_threshold, decided
// in FP32 (an FP64 operation a node was 0.6 % of a query that ends with a
// million nodes): w < floor(t), t = (score / sum + eps) 2^32, is w + 1 <= t, and
// t from 24 bits of score and 1 / sum is off by less than 2^-21 of it (2^-23
// from cutting the score, 2^-24 from each of 1 / sum, eps, w + 1 and three
// roundings), so a difference above 2^-18 of the larger side has the right sign.
// False: not decided.
KP_HD bool draw_decided(uint32_t w, double score, const ScoreSum& s, bool* below) {
  const int hi = hd::high(score);
  if (no_score(hi)) {
    *below = true;
    return true;
  }
  // score inv_m 2^inv_e in two factors: the mantissas' product, a power of two
  const int e = (hi >> 20) - 1023 + s.inv_e;  // at most 1: a score is a part of the sum
  const uint32_t lo = (uint32_t)hd::bits(score);
  const float m = hd::f32(0x3f800000 | (int)((((uint32_t)hi << 3) | (lo >> 29)) & 0x7fffffu));
  const float scale = hd::f32((int)((uint32_t)(e < -126 ? 0 : e + 127) << 23));
  const float t = hd::mul(hd::fma(hd::mul(m, s.inv_m), scale, s.eps32), 4294967296.0f);
  const float w1 = hd::add((float)w, 1.0f);
  *below = w1 < t;
  return e < 64 && fabsf(hd::add(t, -w1)) > hd::mul(fmaxf(t, w1), 3.814697265625e-06f);
}

// The same; one draw in some 100,000 takes the threshold itself.
KP_HD bool draw_accepted(uint32_t w, double score, const ScoreSum& s, double eps) {
  bool below;
  if (draw_decided(w, score, s, &below)) return below;
  return (uint64_t)w < accept_threshold(score, s.sum, s.inv, eps);
}

}  // namespace kp
