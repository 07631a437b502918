// fix64.cuh -- free-space pair terms of the double-precision plans in 64-bit
// integers, with no fewer bits than the FP64 expressions hold.
//
// GB300 issues one FP64 warp instruction per ~19 cycles and SM (measured: 1.05
// TFLOP/s against 78 in single precision), so an FP64 instruction costs as much
// as 76 others, and a pair takes about 47.  In integers it takes about 200:
//   - coordinates as 96-bit fixed point modulo 2^96, in units of 2^-92 of the power
//     of two above the leaf side (near64.cu takes the last five bits of x for the
//     charge): the difference of two points of neighbouring leaves is one integer
//     subtraction, exact for coordinates down to 2^-35 of the leaf side (a double
//     has 53 bits) and to 2^-87 of it below;
//   - a value as 63 bits and an exponent, a product as the upper 64 bits of the
//     128: 1 / r^2 from the single-precision reciprocal and one Newton step of
//     second order, ln r^2 from a table of 512 entries and the series of log1p;
//   - sums over pairs as 128-bit integers, exact.
// A gradient term is good to 2^-54 of |q| / r and a logarithm to 2^-53 of its
// magnitude or of 1 (checked on the CPU; the FP64 expression rounds four times,
// 2^-53 each), and the sums add nothing, where FP64 sums round at every term.
//
// Charges are held relative to the largest: one below 2^-17 of it is as exact as
// one of that size.  A term of it is then off by at most 2^-70 of the largest
// charge over r, r >= 2^-4 leaf sides (closer ones take FP64, fx_cut), which is
// less than the rounding to 53 bits of the largest charge's own field at every
// target within 2^12 leaf sides of it.
//
// The functions compile for the host as well; all but the starting value of the
// reciprocal is integer arithmetic, the same there bit for bit.
#pragma once
#include "ff64.cuh"

FF_HD int fx_clz(uint32_t v) {  // v != 0
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return __builtin_clz(v);
#endif
}
FF_HD int fx_mulhi(int a, int b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int)(((int64_t)a * b) >> 32);
#endif
}
// the upper word of (hi, lo) << s, 0 <= s < 32
FF_HD uint32_t fx_funnel(uint32_t lo, uint32_t hi, int s) {
#ifdef __CUDA_ARCH__
  return __funnelshift_l(lo, hi, s);
#else
  return (uint32_t)(((((uint64_t)hi << 32) | lo) << s) >> 32);
#endif
}

// a 96-bit fixed-point number: v 2^32 + e (v as two's complement)
struct fx96 {
  uint64_t v;
  uint32_t e;
};
// the double v as an integer number of 2^-(s+32), to nearest, modulo 2^96
FF_HD fx96 fx_fixed(double v, int s) {
  uint64_t b;
  memcpy(&b, &v, sizeof b);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return fx96{0, 0};
  const uint64_t m = (b & 0xfffffffffffffull) | (1ull << 52);
  const int sh = ex - 1075 + s + 32;
  uint64_t hi = 0;  // hi 2^64 + lo, modulo 2^128
  uint64_t lo = 0;
  if (sh >= 64) {
    hi = sh < 128 ? m << (sh - 64) : 0;
  } else if (sh >= 0) {
    lo = m << sh;
    hi = sh > 0 ? m >> (64 - sh) : 0;
  } else if (sh >= -54) {
    lo = (m + (1ull << (-sh - 1))) >> -sh;
  }
  if (b >> 63) {
    lo = 0 - lo;
    hi = ~hi + (lo == 0 ? 1 : 0);
  }
  return fx96{(hi << 32) | (lo >> 32), (uint32_t)lo};
}
// a - b
FF_HD fx96 fx_sub(fx96 a, fx96 b) {
  return fx96{a.v - b.v - (a.e < b.e ? 1u : 0u), a.e - b.e};
}

// a b + c.  A shift of a 32-bit number into a 64-bit sum is such a product too:
// the multiplier's pipe has room where the adder's is full.
FF_HD int64_t fx_mad(int a, int b, int64_t c) {
#ifdef __CUDA_ARCH__
  int64_t r;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
#else
  return (int64_t)((uint64_t)((int64_t)a * b) + (uint64_t)c);
#endif
}
FF_HD int fx_hi(int64_t v) { return (int)(v >> 32); }

// a 64-bit integer h 2^32 + 2 l (its lowest bit dropped), so that its halves
// multiply as signed 32-bit numbers
struct fx2 {
  int h, l;
};
FF_HD fx2 fx_halves(int64_t v) { return fx2{fx_hi(v), (int)((uint32_t)v >> 1)}; }
// a b / 2^64, up to 4 units off
FF_HD int64_t fx_mul(fx2 a, fx2 b) {
  const int64_t s = fx_mad(a.l, b.h, (int64_t)a.h * b.l);
  return fx_mad(fx_hi(s), 2, (int64_t)a.h * b.h);
}

// 128-bit sum
struct fx_sum {
  uint64_t lo;
  int64_t hi;
  // + t 2^m, 1 <= m <= 31
  FF_HD void add(int64_t t, int m) {
    const uint32_t tl = (uint32_t)(uint64_t)t, th = (uint32_t)((uint64_t)t >> 32);
    const uint32_t r0 = tl << m, r1 = fx_funnel(tl, th, m);
    const int r2 = (int)th >> (32 - m), r3 = r2 >> 31;
    const uint64_t al = ((uint64_t)r1 << 32) | r0, ah = ((uint64_t)(uint32_t)r3 << 32) | (uint32_t)r2;
#ifdef __CUDA_ARCH__
    asm("add.cc.u64 %0, %0, %2;\n\taddc.u64 %1, %1, %3;" : "+l"(lo), "+l"(hi) : "l"(al), "l"(ah));
#else
    lo += al;
    hi = (int64_t)((uint64_t)hi + ah + (lo < al ? 1 : 0));
#endif
  }
  // the sum times 2^e, rounded once (a sum of magnitude below 2^126)
  FF_HD double value(int e) const {
    uint64_t l = lo, h = (uint64_t)hi;
    const bool neg = hi < 0;
    if (neg) {
      l = 0 - l;
      h = ~h + (l == 0 ? 1 : 0);
    }
    if ((h | l) == 0) return 0.0;
    // to the top of h, the rest as a sticky bit (the conversion rounds to 53)
    int s = 0;
    if (h == 0) {
      h = l;
      l = 0;
      s = 64;
    }
    const uint32_t hh = (uint32_t)(h >> 32);
    const int z = hh ? fx_clz(hh) : 32 + fx_clz((uint32_t)h);
    if (z > 1) {  // z - 1: the conversion is of a signed number
      h = (h << (z - 1)) | (l >> (65 - z));
      l <<= z - 1;
    }
    const int up = z - 1;
    if (up < 0) {
      l |= h & 1;
      h >>= 1;
    }
    h |= l != 0 ? 1 : 0;
    const double d = ldexp((double)(int64_t)h, e + 64 - s - up);
    return neg ? -d : d;
  }
};

// a charge: bits = q 2^(62 - E + drop), E the exponent of the largest (biased: emax),
// drop <= kFxDrop
constexpr int kFxDrop = 17;
struct FxCharge {
  int64_t bits;
  int drop;
};
FF_HD FxCharge fx_charge(double v, int emax) {
  uint64_t b;
  memcpy(&b, &v, sizeof b);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return FxCharge{0, 0};
  const int64_t m = (int64_t)((((b & 0xfffffffffffffull) | (1ull << 52)) << 10));
  const int drop = emax - ex < kFxDrop ? emax - ex : kFxDrop, sh = emax - ex - drop;
  const int64_t q = sh < 63 ? m >> sh : 0;
  return FxCharge{(b >> 63) ? -q : q, drop};
}

// -ln m_i, m_i = 1 + i / 512, or -ln(m_i / 2) from kFfLogTurn on, times 2^60
inline void fx_log_table(int64_t *tab) {  // host
  for (int i = 0; i < kFfLogN; ++i) {
    const long double m = 1.0L + (long double)i / kFfLogN;
    tab[i] = (int64_t)floorl(-logl(i >= kFfLogTurn ? m / 2 : m) * 1152921504606846976.0L + 0.5L);
  }
}

// what depends on the leaf side only: kd, the exponent of the power of two above
// it (the unit of the coordinates' upper 64 bits is 2^(kd-60)), gives the scale
// of the logarithms, 2^(60-v) with v so that they fit, and ln 2 in it; tab: the
// table in it, 2 kd ln 2 added
struct FxScale {
  int v;
  int64_t ln2, base;
  FF_HD int64_t tab(int64_t t) const { return (t >> v) + base; }
};
FF_HD FxScale fx_scale(int kd) {
  FxScale c;
  c.v = 0;
  const int most = 2 * (kd < 0 ? -kd : kd) + 40;  // > |ln r^2| / ln 2 + 2
  while ((10 << c.v) < most && c.v < 12) ++c.v;   // most ln 2 < 8 2^v
  const int64_t ln2 = 799144290325165979;         // 2^60 ln 2
  c.ln2 = (ln2 + ((1ll << c.v) >> 1)) >> c.v;
  c.base = (2 * kd * (ln2 >> 16)) * (1ll << (16 - c.v)) + ((2 * kd * (ln2 & 0xffff)) >> c.v);
  return c;
}

// the larger difference in units of 2^(kd-28), its bits or'ed with the other's;
// below fx_cut a pair is too close for fx_pair: 2^-12 of 2^kd, 2^-4 for the weak
// charges whose lowest bits are cut
FF_HD uint32_t fx_reach(fx96 dx, fx96 dy) {
  const int hx = (int)(dx.v >> 32), hy = (int)(dy.v >> 32);
  return (uint32_t)(hx ^ (hx >> 31)) | (uint32_t)(hy ^ (hy >> 31));
}
FF_HD uint32_t fx_cut(int drop) { return drop < kFxDrop ? 1u << 16 : 1u << 24; }

struct FxSums {
  fx_sum l, x, y;  // sum q ln r^2, sum q dx / r^2, sum q dy / r^2
  FF_HD void clear() { l = x = y = fx_sum{0, 0}; }
  // the values for charges of largest biased exponent emax
  FF_HD double log_sum(int emax, const FxScale &c) const { return l.value(emax - 1023 + c.v - 76); }
  FF_HD double gx(int emax, int kd) const { return x.value(emax - 1023 - kd - 77); }
  FF_HD double gy(int emax, int kd) const { return y.value(emax - 1023 - kd - 77); }
};

// 1 / f to about 2^-23; NUDGE of the host checks moves it by that many ulps
FF_HD float fx_rcp(float f, int nudge) {
#ifdef __CUDA_ARCH__
  return ff_rcp_approx(f);
#else
  return ff_from(ff_bits(1.0f / f) + (uint32_t)nudge);
#endif
}
FF_HD uint32_t fx_to_uint(float f) {  // to nearest
#ifdef __CUDA_ARCH__
  return __float2uint_rn(f);
#else
  return (uint32_t)lrintf(f);
#endif
}

// The terms of a charge q at the difference (dx, dy) added to the sums; reach:
// fx_reach of it, fx_cut .. 2^30 - 1; tab: fx_log_table by FxScale::tab.
FF_HD void fx_pair(FxSums &a, fx96 dx, fx96 dy, uint32_t reach, int64_t qbits, int drop,
                   const FxScale &c, const int64_t *tab, int nudge = 0) {
  // x, y = the differences times 2^s (s = 1 .. 14), the larger with 63 bits
  const int s = fx_clz(reach) - 1;
  const fx2 x{(int)fx_funnel((uint32_t)dx.v, (uint32_t)(dx.v >> 32), s),
              (int)(fx_funnel(dx.e, (uint32_t)dx.v, s) >> 1)};
  const fx2 y{(int)fx_funnel((uint32_t)dy.v, (uint32_t)(dy.v >> 32), s),
              (int)(fx_funnel(dy.e, (uint32_t)dy.v, s) >> 1)};
  // R = (x^2 + y^2) / 2^64 to 5 units, 2^60 .. 2^63 (unsigned)
  const int64_t cross = fx_mad(x.h, x.l, (int64_t)y.h * y.l);
  const uint64_t R =
      (uint64_t)fx_mad(fx_hi(cross), 4, fx_mad(x.h, x.h, (int64_t)y.h * y.h));
  const float cf = fx_rcp((float)(uint32_t)(R >> 32), nudge);
  // C = 2^122 / R: c0 = 2^84 / R to 2^-21.2, e = R c0 - 2^84 (exact, |e| < 2^63),
  // C = 2^38 c0 (1 - e / 2^84 + (e / 2^84)^2)
  const uint32_t c0 = fx_to_uint(cf * 4503599627370496.0f /* 2^52 */);
  const uint64_t e = R * c0;
  const int eh = (int)(e >> 32);
  const int64_t U = fx_mad(eh, (int)c0, (int64_t)(((uint64_t)(uint32_t)e * c0) >> 32));
  const int e2 = fx_mulhi(eh, eh);
  const int64_t C = (int64_t)((uint64_t)(c0 << 6) << 32) - (U >> 14) + (fx_mulhi((int)c0, e2) >> 2);
  // gradient terms q C x / 2^128
  const fx2 q = fx_halves(qbits), w = fx_halves(fx_mul(q, fx_halves(C)));
  const int m = kFxDrop + s - drop;
  a.x.add(fx_mul(w, x), m);
  a.y.add(fx_mul(w, y), m);
  // ln R = k ln 2 + tab + log1p(t): c' = cf rounded to 9 bits, t = R c' - 1 as
  // 2^72 t, exact (|t| < 2^-9.9)
  const uint32_t cb = ff_bits(cf) + (1u << (22 - kFfLogBits));
  const uint32_t i = (cb >> (23 - kFfLogBits)) & (kFfLogN - 1);
  const int z = (int)(cb >> 23) - 96;  // 0 .. 3
  const int64_t t = (int64_t)(R * (uint64_t)((kFfLogN + i) << z));
  const int th = fx_hi(t), tl = (int)((uint32_t)t >> 1);
  // t^3 (1/3 - t/4 + t^2/5) times 2^56
  const int u = fx_mulhi(th, th);  // 2^48 t^2
  const int cub = fx_mulhi(fx_mulhi(u, th), 1431655765 - (th >> 10) + (fx_mulhi(u, 858993459) >> 16));
  // 2^80 (t^2 - 2 of that)
  const int64_t t2 = fx_mad(cub, -(1 << 25), fx_mad(fx_mulhi(th, tl), 4, (int64_t)th * th));
  const uint32_t eb = (cb + (0x800000u - ((uint32_t)kFfLogTurn << (23 - kFfLogBits)))) >> 23;
  const int k = 103 - (int)eb - 2 * s;  // -25 .. 5
  const int64_t L = tab[i] + (t >> (12 + c.v)) - (t2 >> (21 + c.v)) + (int64_t)k * c.ln2;
  a.l.add(fx_mul(q, fx_halves(L)), kFxDrop + 1 - drop);
}
