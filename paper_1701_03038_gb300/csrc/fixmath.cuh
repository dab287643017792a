// fixmath.cuh -- the exponential and the logarithm of the log-sums, and the
// float conversions around them, in integer arithmetic.
//
// This part has one float64 unit per 64 float32 ones: a warp's float64
// instruction holds its scheduler for 64 cycles, and a float64 exp or log is
// some 30 of them.  The log-sums need neither's range: their terms are
// exp(v - max) as 2^-40 fixed-point integers, and their sums are integers of
// at least 2^40.  So the argument is taken apart as an integer, reduced
// against a table (the table-driven method of P. T. P. Tang, ACM
// TOMS 15 (1989) and 16 (1990)) and finished with a short polynomial in 32-
// and 64-bit products.  Errors, against 80-bit arithmetic over the whole
// range: the term is within 0.53 of a unit of 2^-40 (0.50 is its rounding),
// the logarithm within 1e-15 plus half a unit of the float64 result.
#pragma once

#include <math.h>
#include <stdint.h>
#include <string.h>

#include "fixmath_tables.cuh"

namespace fstgpu {

#ifdef __CUDACC__
#define FX_FN __device__ __forceinline__
FX_FN uint64_t fx_mulhi(uint64_t a, uint64_t b) { return __umul64hi(a, b); }
FX_FN int64_t fx_mulhi_s(int64_t a, int64_t b) { return __mul64hi(a, b); }
FX_FN uint32_t fx_mulhi32(uint32_t a, uint32_t b) { return __umulhi(a, b); }
FX_FN int fx_clz(uint64_t x) { return __clzll((long long)x); }
FX_FN uint64_t fx_bits(double x) { return (uint64_t)__double_as_longlong(x); }
FX_FN double fx_double(uint64_t u) { return __longlong_as_double((long long)u); }
FX_FN uint32_t fx_bits32(float x) { return __float_as_uint(x); }
FX_FN float fx_float(uint32_t u) { return __uint_as_float(u); }
FX_FN uint64_t fx_table(const uint64_t* t, int i) { return __ldg((const unsigned long long*)t + i); }
FX_FN int32_t fx_round32(float x) { return __float2int_rn(x); }
#else  // the host's copy, for error measurements
#define FX_FN inline
FX_FN uint64_t fx_mulhi(uint64_t a, uint64_t b) { return (uint64_t)(((unsigned __int128)a * b) >> 64); }
FX_FN int64_t fx_mulhi_s(int64_t a, int64_t b) { return (int64_t)(((__int128)a * b) >> 64); }
FX_FN uint32_t fx_mulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((uint64_t)a * b) >> 32); }
FX_FN int fx_clz(uint64_t x) { return __builtin_clzll(x); }
FX_FN uint64_t fx_bits(double x) { uint64_t u; memcpy(&u, &x, 8); return u; }
FX_FN double fx_double(uint64_t u) { double x; memcpy(&x, &u, 8); return x; }
FX_FN uint32_t fx_bits32(float x) { uint32_t u; memcpy(&u, &x, 4); return u; }
FX_FN float fx_float(uint32_t u) { float x; memcpy(&x, &u, 4); return x; }
FX_FN uint64_t fx_table(const uint64_t* t, int i) { return t[i]; }
FX_FN int32_t fx_round32(float x) { return (int32_t)lrintf(x); }
#endif

// round(exp(x) 2^40) for a finite x <= 0.
FX_FN uint64_t fx_exp40(double x) {
  const uint64_t u = fx_bits(x);
  const int ex = (int)((u >> 52) & 0x7ff) - 1023;
  if (ex < -58) return 1ull << 40;
  if (ex > 4) return 0ull;
  // |x| in 2^-58 (below 2^5)
  const uint64_t m = (u & 0xfffffffffffffull) | 0x10000000000000ull;
  const uint64_t d = ex >= -6 ? m << (ex + 6) : m >> (-6 - ex);
  // |x| = n ln2 / 128 + r, 0 <= r < 0.0055
  const uint32_t n = (uint32_t)(((d >> 31) * 48408412ull) >> 45);
  const uint64_t r = d - (uint64_t)n * FX_LN2_128;
  if (n >= 41u * 128u) return 0ull;
  // w = 1 - exp(-r) = r - r^2 (1/2 - r (1/6 - r (1/24 - r / 120)))
  const uint32_t r39 = (uint32_t)(r >> 19);
  uint32_t t = 178956971u - (fx_mulhi32(r39, 35791394u) >> 7);  // 1/24, 1/120 in 2^-32
  t = 715827883u - (fx_mulhi32(r39, t) >> 7);                   // 1/6
  t = 2147483648u - (fx_mulhi32(r39, t) >> 7);                  // 1/2
  const uint64_t w = r - ((uint64_t)fx_mulhi32(fx_mulhi32(r39, r39), t) << 12);
  const uint64_t T = fx_table(FX_EXP, (int)(n & 127u));  // 2^(-i/128) in 2^-63
  const uint64_t y = T - 2ull * fx_mulhi(T, w << 5);
  const int sh = 23 + (int)(n >> 7);
  return (y + (1ull << (sh - 1))) >> sh;
}

// log x in 2^-58, x in [2^63, 2^64) standing for [1, 2).
FX_FN int64_t fx_log58(uint64_t x) {
  const int i = (int)(x >> 55) & 255;
  // x c with c about 1 / x: 1 + d, |d| < 2^-9
  const int64_t d = (int64_t)(fx_mulhi(x, fx_table(FX_INV, i)) - (1ull << 63));  // in 2^-63
  const int64_t d2 = fx_mulhi_s(d, d);                                         // d^2 in 2^-62
  const float f = (float)(int32_t)(d >> 24) * 1.8189894035458565e-12f;           // d (2^-39)
  const float rest = f * f * f * (0.33333333f - f * (0.25f - f * 0.2f));
  return (int64_t)fx_table(FX_LOG, i) + (d >> 5) - (d2 >> 5) + (int64_t)fx_round32(rest * 288230376151711744.f);  // 2^58
}

// m + log(s 2^-40), s >= 2^40.
FX_FN double fx_add_log40(double m, uint64_t s) {
  const int z = fx_clz(s);
  const int64_t l = fx_log58(s << z) + (int64_t)(23 - z) * FX_LN2_58;
  return m + (double)l * 3.469446951953614e-18;  // 2^-58
}

// A float32 as float64.
FX_FN double fx_widen(float x) {
  const uint32_t u = fx_bits32(x), e = (u >> 23) & 255u;
  if (e == 0u) return (u << 1) ? (double)x : fx_double((uint64_t)u << 32);
  uint32_t hi = (u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u);
  if (e == 255u) hi |= 0x7ff00000u;
  return fx_double(((uint64_t)hi << 32) | (uint64_t)(u << 29));
}
// A float64 rounded to float32 (to nearest, ties to even).
FX_FN float fx_narrow(double x) {
  const uint64_t u = fx_bits(x);
  const uint32_t e = (uint32_t)(u >> 52) & 0x7ffu;
  if (e < 897u || e > 1149u) return (u << 1) ? (float)x : fx_float((uint32_t)(u >> 32));
  const uint64_t a = (u & 0x7fffffffffffffffull) - (896ull << 52);
  const uint32_t r = (uint32_t)((a + 0xfffffffull + ((a >> 29) & 1ull)) >> 29);
  return fx_float((uint32_t)(u >> 63 << 31) | r);
}

}  // namespace fstgpu
