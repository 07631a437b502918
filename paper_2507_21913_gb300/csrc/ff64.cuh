// ff64.cuh -- arithmetic of more than single precision on the single-precision
// pipe: a value as an unevaluated sum h + l of two floats, about 48 bits, with the
// error-free sum and product of Dekker and Knuth.  GB300 issues one FP64 warp
// instruction per ~19 cycles and SM, so an FP64 instruction costs as much as 76
// single-precision ones.  For values that are rounded to single precision in the
// end (mirror_ff.cuh); the pairs of double-precision plans need more bits and take
// integers (fix64.cuh).  The conversions from fixed point and the three-float sum
// belong to the same arithmetic and are checked with it.
//
// The functions compile for the host as well (with the same roundings), so
// that the arithmetic is checked on the CPU.
#pragma once
#include <math.h>
#include <stdint.h>
#include <string.h>

#ifdef __CUDACC__
#define FF_HD __host__ __device__ __forceinline__
#else
#define FF_HD inline
#endif

// single operations that the compiler may not contract into one another
FF_HD float ff_add(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fadd_rn(a, b);
#else
  volatile float s = a + b;
  return s;
#endif
}
FF_HD float ff_mul(float a, float b) {
#ifdef __CUDA_ARCH__
  return __fmul_rn(a, b);
#else
  volatile float s = a * b;
  return s;
#endif
}
FF_HD float ff_sub(float a, float b) { return ff_add(a, -b); }
FF_HD float ff_fma(float a, float b, float c) { return fmaf(a, b, c); }
FF_HD uint32_t ff_bits(float v) {
  uint32_t u;
  memcpy(&u, &v, sizeof u);
  return u;
}
FF_HD float ff_from(uint32_t u) {
  float v;
  memcpy(&v, &u, sizeof v);
  return v;
}
// an approximation of 1 / x to about 2^-23 (refined by its users)
FF_HD float ff_rcp_approx(float x) {
#ifdef __CUDA_ARCH__
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
#else
  return 1.0f / x;
#endif
}

struct ff {
  float h, l;
};

// s + e = a + b exactly (Knuth); ff_quick: the same for |a| >= |b| or a = 0
FF_HD ff ff_two_sum(float a, float b) {
  const float s = ff_add(a, b), bb = ff_sub(s, a);
  return ff{s, ff_add(ff_sub(a, ff_sub(s, bb)), ff_sub(b, bb))};
}
FF_HD ff ff_quick(float a, float b) {
  const float s = ff_add(a, b);
  return ff{s, ff_sub(b, ff_sub(s, a))};
}
// a b exactly
FF_HD ff ff_two_prod(float a, float b) {
  const float p = ff_mul(a, b);
  return ff{p, ff_fma(a, b, -p)};
}
// the product of two pairs, not renormalised (l stays below 2^-22 of h)
FF_HD ff ff_prod(ff a, ff b) {
  ff p = ff_two_prod(a.h, b.h);
  p.l = ff_fma(a.h, b.l, ff_fma(a.l, b.h, p.l));
  return p;
}

// a running sum as three floats: a and b take exact sums, c what remains
struct ff_sum3 {
  float a, b, c;
  FF_HD void add(ff t) {
    const ff s = ff_two_sum(a, t.h);
    const ff r = ff_two_sum(b, ff_add(t.l, s.l));
    a = s.h;
    b = r.h;
    c = ff_add(c, r.l);
  }
  FF_HD double value() const { return (double)a + ((double)b + (double)c); }
};

// the double v as an integer number of 2^-s (to nearest, ties up), modulo 2^64
FF_HD int64_t ff_fixed(double v, int s) {
  uint64_t b;
  memcpy(&b, &v, sizeof b);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e == 0) return 0;
  const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
  const int sh = e - 1075 + s;
  uint64_t r;
  if (sh >= 64) r = 0;
  else if (sh >= 0) r = m << sh;
  else if (sh >= -54) r = (m + (1ull << (-sh - 1))) >> -sh;
  else r = 0;
  return (int64_t)((b >> 63) ? 0 - r : r);
}

// a difference D (|D| < 2^62) of fixed-point coordinates, in units of 2^37,
// as a normalised pair: three non-overlapping pieces of D, each made a float
// by the exponent of 2^23 (or 1.5 2^23 for the signed one)
FF_HD ff ff_from_fixed(int64_t D) {
  const uint32_t lo = (uint32_t)(uint64_t)D;
  const int32_t hi = (int32_t)(D >> 32);
  const float f1 = ff_sub(ff_from((uint32_t)(0x4B400000 + (hi >> 8))), 12582912.0f);  // 2^40
  const uint32_t mid = (uint32_t)((uint64_t)D >> 17);
  const float f2 = ff_sub(ff_from(0x4B000000u | (mid & 0x7fffffu)), 8388608.0f);  // 2^17
  const float f3 = ff_sub(ff_from(0x4B000000u | (lo & 0x1ffffu)), 8388608.0f);    // 1
  // units of 2^37
  const float t = ff_mul(f1, 8.0f), u = ff_mul(f2, 9.5367431640625e-07f /* 2^-20 */);
  const ff a = ff_quick(t, u);
  return ff_quick(a.h, ff_fma(f3, 7.275957614183426e-12f /* 2^-37 */, a.l));
}

// dx^2 + dy^2
FF_HD ff ff_norm2(ff x, ff y) {
  ff a = ff_two_prod(x.h, x.h), b = ff_two_prod(y.h, y.h);
  a.l = ff_fma(ff_add(x.h, x.h), x.l, a.l);
  b.l = ff_fma(ff_add(y.h, y.h), y.l, b.l);
  const ff s = ff_two_sum(a.h, b.h);
  return ff_quick(s.h, ff_add(s.l, ff_add(a.l, b.l)));
}

// 1 / r; c: an approximation of 1 / r.h
FF_HD ff ff_recip(ff r, float c) {
  // the float nearest to 1 / r, then the remainder 1 - r c1 (below 2^-23)
  float a = ff_mul(r.h, c);
  float e = ff_fma(-r.l, c, ff_sub(ff_sub(1.0f, a), ff_fma(r.h, c, -a)));
  const float c1 = ff_fma(c, e, c);
  a = ff_mul(r.h, c1);
  e = ff_fma(-r.l, c1, ff_sub(ff_sub(1.0f, a), ff_fma(r.h, c1, -a)));
  return ff{c1, ff_mul(c1, e)};
}

// Natural logarithm, ln r = k ln 2 + m with |m| < 0.37, k an integer.  c' = an
// approximation of 1 / r of kFfLogBits mantissa bits; with t = r c' - 1 (exact
// products, |t| <= 2^-10) ln r = -ln c' + log1p(t), ln c' from a table over its
// mantissa and its exponent.  Entry i of the table: -ln m_i, m_i = 1 + i / 512,
// or -ln(m_i / 2) from kFfLogTurn on, so that the entries lie around 0.  k is
// left apart: the caller sums q k and q m, so that the rounding of the sums
// follows |m| and not |ln r| (an absolute error of about 2^-48).
constexpr int kFfLogBits = 9, kFfLogN = 1 << kFfLogBits, kFfLogTurn = 212;
inline void ff_log_table(ff *tab) {  // host
  for (int i = 0; i < kFfLogN; ++i) {
    const long double m = 1.0L + (long double)i / kFfLogN;
    const long double v = -logl(i >= kFfLogTurn ? m / 2 : m);
    tab[i].h = (float)v;
    tab[i].l = (float)(v - (long double)tab[i].h);
  }
}
// c: an approximation of 1 / r.h; ebias: subtracted from the exponent of r
// (|ebias| < 4000: any side a double can hold)
FF_HD ff ff_log(ff r, float c, const ff *tab, int ebias, float &k) {
  const uint32_t cb = (ff_bits(c) + (1u << (22 - kFfLogBits))) & ~((1u << (23 - kFfLogBits)) - 1u);
  const float cr = ff_from(cb);
  const ff T = tab[(cb >> (23 - kFfLogBits)) & (kFfLogN - 1)];
  // -(exponent of c'), one less from kFfLogTurn on
  const uint32_t eb = (cb + (0x800000u - ((uint32_t)kFfLogTurn << (23 - kFfLogBits)))) >> 23;
  k = ff_sub((float)(8388608 + 127 + 4096),
             ff_from(0x4B000000u | (eb + (uint32_t)(ebias + 4096))));
  const float a = ff_mul(r.h, cr);
  const float th = ff_sub(a, 1.0f);
  const float tl = ff_fma(r.l, cr, ff_fma(r.h, cr, -a));
  // log1p(t) = t - t^2/2 + t^3 (1/3 - t/4 + t^2/5); a table entry is 0 or at
  // least 2^-9.5 in magnitude
  const float h2 = ff_mul(-0.5f, th);
  const ff m = ff_two_prod(h2, th);
  const float cub = ff_mul(ff_mul(ff_mul(-2.0f, m.h), th),
                           ff_fma(th, ff_fma(th, 0.2f, -0.25f), 0.333333343f));
  // the low part's share of the higher terms, tl (-th + th^2 - tl/2)
  const float u = ff_fma(-0.5f, tl, ff_fma(th, th, -th));
  const ff s1 = ff_quick(T.h, th), s2 = ff_quick(s1.h, m.h);
  const float lo = ff_add(ff_add(T.l, ff_add(s1.l, s2.l)),
                          ff_add(tl, ff_fma(u, tl, ff_add(m.l, cub))));
  return ff_quick(s2.h, lo);
}

// a double as a pair: h rounded toward zero to 24 bits, l the other 29 rounded
// to 24; the exponent is reduced by `down`, and what then falls below 2^-90 is
// zero (the caller scales by the largest value)
FF_HD ff ff_split_scaled(double v, int down) {
  uint64_t b;
  memcpy(&b, &v, sizeof b);
  const int e = (int)((b >> 52) & 0x7ff) - 1023 - down;
  if (((b >> 52) & 0x7ff) == 0 || e < -90) return ff{0.0f, 0.0f};
  const uint32_t sign = (uint32_t)(b >> 63) << 31;
  const uint32_t top = (uint32_t)((b & 0xfffffffffffffull) >> 29);  // 23 bits
  const uint32_t rest = (uint32_t)(b & 0x1fffffffull);              // 29 bits
  const float h = ff_from(sign | ((uint32_t)(e + 127) << 23) | top);
  const float sc = ff_from((uint32_t)(e - 30 + 127) << 23);  // 2^(e-30): >= 2^-120
  const float l = ff_mul((float)(int32_t)rest, sc);          // in units of 4 2^(e-52+...)
  return ff{h, (sign ? -l : l) * 2.384185791015625e-07f /* 2^-22 */};
}
