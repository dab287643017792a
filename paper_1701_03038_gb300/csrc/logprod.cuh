// logprod.cuh -- the exponentials and the logarithm of a product of log-weight
// matrices in the linear domain (prefix.cu), in float32.
//
// An entry is r + c + log sum_k exp(A - r) exp(B - c) with r and c the scales
// of its row and column.  r + c may be far larger than the entry, and a string
// of 1,000 symbols adds up the errors of 999 products, so that a bias of a
// tenth of a rounding shows: differences and sums that are not exact carry
// their rounding errors along, and the exponential is rounded evenly (CUDA's
// expf is 6e-9 to 1.1e-8 too large on average, which an entry would have
// twice).
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

namespace fstgpu {

#ifdef __CUDACC__
#define LP_FN __device__ __forceinline__
LP_FN float lp_add(float a, float b) { return __fadd_rn(a, b); }
LP_FN float lp_sub(float a, float b) { return __fsub_rn(a, b); }
LP_FN float lp_mul(float a, float b) { return __fmul_rn(a, b); }
LP_FN uint32_t lp_bits(float x) { return __float_as_uint(x); }
LP_FN float lp_float(uint32_t u) { return __uint_as_float(u); }
#else  // the host's copy, for error measurements
#define LP_FN inline
LP_FN float lp_add(float a, float b) { volatile float x = a + b; return x; }
LP_FN float lp_sub(float a, float b) { volatile float x = a - b; return x; }
LP_FN float lp_mul(float a, float b) { volatile float x = a * b; return x; }
LP_FN uint32_t lp_bits(float x) { uint32_t u; memcpy(&u, &x, 4); return u; }
LP_FN float lp_float(uint32_t u) { float x; memcpy(&x, &u, 4); return x; }
#endif

// log 2 in 12 bits, whose multiples below 2^12 are exact, and the rest.
#define LP_LN2_HI 0.693115234375f
#define LP_LN2_LO 3.194618494530942e-05f

// The rounded sum and its error: a + b = s + e exactly (Knuth, TAOCP 2, 4.2.2).
struct Sum2 {
  float s, e;
};
LP_FN Sum2 add2(float a, float b) {
  const float s = lp_add(a, b), t = lp_sub(s, a);
  return Sum2{s, lp_add(lp_sub(a, lp_sub(s, t)), lp_sub(b, t))};
}

// A row's or column's scale: its largest entry, rounded up to a quarter where
// that is exact.  Differences and sums with such scales mostly are, too.
constexpr float SCALE_MAX = 1048576.f;  // 2^20
LP_FN float scale_of(float m) { return fabsf(m) < SCALE_MAX ? ceilf(4.f * m) * 0.25f : m; }

// exp(x), x <= 0; 0 below 2^-126, and for NaN.  x = k log 2 + r with |r| <=
// 0.35, k log 2 taken off in two parts, the first exactly (Cody and Waite,
// Software Manual for the Elementary Functions, 1980), then the Taylor series
// of exp(r).  k is rounded by an addition that leaves it in the low bits.
LP_FN float exp_neg(float x) {
  if (!(x >= -87.3f)) return 0.f;
  const float kb = fmaf(x, 1.44269504f, 12582912.f), k = lp_sub(kb, 12582912.f);  // 1.5 * 2^23
  const float r = fmaf(k, -LP_LN2_LO, fmaf(k, -LP_LN2_HI, x));
  float q = 1.f / 40320.f;
  q = fmaf(q, r, 1.f / 5040.f);
  q = fmaf(q, r, 1.f / 720.f);
  q = fmaf(q, r, 1.f / 120.f);
  q = fmaf(q, r, 1.f / 24.f);
  q = fmaf(q, r, 1.f / 6.f);
  q = fmaf(q, r, 0.5f);
  const float y = lp_add(1.f, fmaf(lp_mul(r, r), q, r));
  return lp_float(lp_bits(y) + (lp_bits(kb) << 23));  // (k >= -126, and y >= 1 there)
}

// exp(x - m), x <= m, m a scale: within the roundings of the exponential and
// of the product, whatever the sizes of x and m.  (Below a scale of at most 0
// the difference is exact: both are multiples of x's last place, or it is so
// large that the exponential is 0.)
LP_FN float exp_below(float x, float m) {
  if (m <= 0.f && m > -SCALE_MAX) return exp_neg(lp_sub(x, m));
  const Sum2 d = add2(x, -m);
  const float y = exp_neg(d.s);
  return y == 0.f ? 0.f : fmaf(y, d.e, y);  // (x or m infinite: 0)
}

// r + c + log x, r and c scales, x normal and positive, rounded about once:
// log x = k log 2 + log f with f in [0.7, 1.42).
LP_FN float add_log(float r, float c, float x) {
  const uint32_t u = lp_bits(x);
  float f = lp_float((u & 0x7fffffu) | 0x3f800000u), k = (float)((int32_t)(u >> 23) - 127);
  if (f > 1.41f) {
    f *= 0.5f;
    k += 1.f;
  }
  const float low = fmaf(k, LP_LN2_LO, logf(f));
  // (multiples of 2^-12 below 2^12: their sums are exact)
  if (fabsf(r) < 1024.f && fabsf(c) < 1024.f) return lp_add(lp_add(lp_add(r, c), lp_mul(k, LP_LN2_HI)), low);
  const Sum2 a = add2(r, c), b = add2(a.s, lp_mul(k, LP_LN2_HI));
  if (isinf(b.s)) return b.s;
  return lp_add(b.s, lp_add(lp_add(a.e, b.e), low));
}

}  // namespace fstgpu
