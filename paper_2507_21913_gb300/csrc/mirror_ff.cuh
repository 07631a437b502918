// mirror_ff.cuh -- J_0 and J_1 of the reaction pairs close to the boundary in
// float pairs (ff64.cuh): the double-precision option of single-precision plans
// (HPFMM_MIXED), whose pair values are rounded to single precision.  GB300 takes
// 76 issue slots for an FP64 instruction, about 210 of which the FP64 form of a
// pair needs (16000 slots); this form takes about 900 (550 for real kappa).
//
// For |P| <= 1/8, P = kappa (Y -+ i X), with Q = P^2 and C = P^3
//   e^{-P} - 1 = -P + Q/2 - C/6 + Q v,   sum P^k/(k k!) = P + Q/4 + C/18 + Q w,
// v and w (below 2^-10) by their series in single precision, the rest in pairs;
// J_0 = e^{-P} [i pi - gamma - Log P - sum], J_1 = 1 + P J_0.  Relative error
// below 2^-36 of J_0 and J_1 (checked on the CPU), 2^-12 of the rounding that follows.
#pragma once
#include "ff64.cuh"

struct fc {  // complex pair
  ff x, y;
};
FF_HD ff ff_plus(ff a, ff b) {
  const ff s = ff_two_sum(a.h, b.h);
  return ff_quick(s.h, ff_add(s.l, ff_add(a.l, b.l)));
}
FF_HD ff ff_neg(ff a) { return ff{-a.h, -a.l}; }
FF_HD ff ff_times(ff a, float b) {
  const ff p = ff_two_prod(a.h, b);
  return ff_quick(p.h, ff_fma(a.l, b, p.l));
}
FF_HD ff ff_mult(ff a, ff b) {
  const ff p = ff_prod(a, b);
  return ff_quick(p.h, p.l);
}
FF_HD ff ff_scale(ff a, float p2) { return ff{a.h * p2, a.l * p2}; }  // p2 a power of two
FF_HD fc fc_plus(fc a, fc b) { return fc{ff_plus(a.x, b.x), ff_plus(a.y, b.y)}; }
FF_HD fc fc_mult(fc a, fc b) {
  return fc{ff_plus(ff_mult(a.x, b.x), ff_neg(ff_mult(a.y, b.y))),
            ff_plus(ff_mult(a.x, b.y), ff_mult(a.y, b.x))};
}
FF_HD ff ff_of(double v) {
  const float h = (float)v;
  return ff{h, (float)(v - (double)h)};
}

// atan2(|x|, y) for x, y >= 0: the multiple a_i = i pi/512 of pi/512 nearest to
// it, then atan z = z - z^3/3 + z^5/5, z = tan of the rest (below 2^-8) from the
// table's sine and cosine.  near: a single-precision value of the angle.
constexpr int kFfAng = 257;
struct FfAngle {
  ff a, s, c;
};
inline void ff_angle_table(FfAngle *t) {  // host
  for (int i = 0; i < kFfAng; ++i) {
    const long double a = 3.14159265358979323846264338327950288L * i / 512;
    const long double v[3] = {a, sinl(a), cosl(a)};
    ff *o[3] = {&t[i].a, &t[i].s, &t[i].c};
    for (int e = 0; e < 3; ++e) {
      o[e]->h = (float)v[e];
      o[e]->l = (float)(v[e] - (long double)o[e]->h);
    }
  }
}
FF_HD ff ff_angle(float ax, float y, float near, const FfAngle *tab) {
  int i = (int)(near * 162.97466172610082f + 0.5f);
  i = i < 0 ? 0 : (i > kFfAng - 1 ? kFfAng - 1 : i);
  const FfAngle t = tab[i];
  const ff num = ff_plus(ff_times(t.c, ax), ff_neg(ff_times(t.s, y)));
  const ff den = ff_plus(ff_times(t.s, ax), ff_times(t.c, y));
  const ff z = ff_mult(num, ff_recip(den, ff_rcp_approx(den.h)));
  const float z2 = z.h * z.h;
  const float corr = z.h * z2 * ff_fma(z2, 0.2f, -0.333333343f);
  return ff_plus(t.a, ff_quick(z.h, ff_add(z.l, corr)));
}

// kappa and its logarithm in pairs
struct KappaFF {
  ff kr, ki, lk, ak;
  bool real;
};

// c[0] + c[1] z + ... + c[N-1] z^(N-1) in single precision
template <int N>
FF_HD void ff_tail(const float (&c)[N], float x, float y, float &ox, float &oy) {
  ox = c[N - 1];
  oy = 0.0f;
#ifdef __CUDACC__
#pragma unroll
#endif
  for (int k = N - 2; k >= 0; --k) {
    const float t = ff_fma(ox, x, ff_fma(-oy, y, c[k]));
    oy = ff_fma(ox, y, oy * x);
    ox = t;
  }
}

// e^{-P} - 1 and sum_{k>=1} P^k/(k k!)
FF_HD void ff_exp_sum(fc P, fc &E1, fc &S) {
  const ff xy = ff_mult(P.x, P.y);
  const fc Q{ff_plus(ff_mult(P.x, P.x), ff_neg(ff_mult(P.y, P.y))), ff_scale(xy, 2.0f)};
  const fc C = fc_mult(Q, P);
  const float ce[6] = {1.0f / 24, -1.0f / 120, 1.0f / 720, -1.0f / 5040, 1.0f / 40320,
                       -1.0f / 362880};
  const float cs[6] = {1.0f / 96, 1.0f / 600, 1.0f / 4320, 1.0f / 35280, 1.0f / 322560,
                       1.0f / 3265920};
  float ex, ey, sx, sy;
  ff_tail<6>(ce, P.x.h, P.y.h, ex, ey);
  ff_tail<6>(cs, P.x.h, P.y.h, sx, sy);
  // Q^2 in single precision: Q v = Q^2 (1/24 - P/120 + ...)
  const float qx = Q.x.h, qy = Q.y.h, fx = qx * qx - qy * qy, fy = 2.0f * qx * qy;
  const ff sixth{0.16666667163372039794921875f, -4.967053879312289e-09f};
  const ff eighteenth{0.055555555969476699829101562f, -4.1392114735749885e-10f};
  E1.x = ff_plus(ff_plus(ff_neg(P.x), ff_scale(Q.x, 0.5f)),
                 ff_plus(ff_neg(ff_mult(C.x, sixth)), ff{fx * ex - fy * ey, 0.0f}));
  E1.y = ff_plus(ff_plus(ff_neg(P.y), ff_scale(Q.y, 0.5f)),
                 ff_plus(ff_neg(ff_mult(C.y, sixth)), ff{fx * ey + fy * ex, 0.0f}));
  S.x = ff_plus(ff_plus(P.x, ff_scale(Q.x, 0.25f)),
                ff_plus(ff_mult(C.x, eighteenth), ff{fx * sx - fy * sy, 0.0f}));
  S.y = ff_plus(ff_plus(P.y, ff_scale(Q.y, 0.25f)),
                ff_plus(ff_mult(C.y, eighteenth), ff{fx * sy + fy * sx, 0.0f}));
}

// J_0 and J_1 = 1 + P J_0 from the parts: B = i pi - gamma - Log P - sum
FF_HD void ff_j01(fc P, fc E1, fc B, fc &J0, fc &J1) {
  J0 = fc_plus(B, fc_mult(E1, B));
  J1 = fc_mult(P, J0);
  J1.x = ff_plus(J1.x, ff{1.0f, 0.0f});
}

// u and its gradient for a unit charge (image and reaction), v[6] as MirrorVal,
// |P| <= 1/8, s2 = X^2 + Y^2 >= 2^-80; near: atan2(|X|, Y) in single precision
FF_HD void ff_mirror(float X, float Y, const KappaFF &K, float near, const ff *ltab,
                     const FfAngle *atab, float (&v)[6]) {
  const ff s2 = ff_norm2(ff{X, 0.0f}, ff{Y, 0.0f});
  const float c = ff_rcp_approx(s2.h);
  float k;
  const ff m = ff_log(s2, c, ltab, 0, k);
  ff ln = ff_two_prod(k, 0.693147182464599609375f);
  ln = ff_plus(ff_quick(ln.h, ff_fma(k, -1.9046542121259336e-09f, ln.l)), m);
  const ff inv = ff_recip(s2, c);
  ff th = ff_angle(fabsf(X), Y, near, atab);
  if (X < 0.0f) th = ff_neg(th);
  const ff half_ln = ff_scale(ln, 0.5f);
  const ff g = ff_neg(ff_plus(ff_plus(K.lk, half_ln), ff{0.577215671539306640625f, -6.637773886097875e-09f}));
  const ff pi{3.1415927410125732421875f, -8.742277657347586e-08f};
  const ff ry = ff_times(K.kr, Y), rx = ff_times(K.kr, X);
  fc Pp{ry, ff_neg(rx)}, Pm{ry, rx};
  if (!K.real) {
    const ff iy = ff_times(K.ki, Y), ix = ff_times(K.ki, X);
    Pp = fc{ff_plus(ry, ix), ff_plus(iy, ff_neg(rx))};
    Pm = fc{ff_plus(ry, ff_neg(ix)), ff_plus(iy, rx)};
  }
  fc Ep, Sp, Em, Sm;
  ff_exp_sum(Pp, Ep, Sp);
  if (K.real) {
    Em = fc{Ep.x, ff_neg(Ep.y)};
    Sm = fc{Sp.x, ff_neg(Sp.y)};
  } else {
    ff_exp_sum(Pm, Em, Sm);
  }
  const ff pa = ff_plus(pi, ff_neg(K.ak));
  const fc Bp{ff_plus(g, ff_neg(Sp.x)), ff_plus(ff_plus(pa, th), ff_neg(Sp.y))};
  const fc Bm{ff_plus(g, ff_neg(Sm.x)), ff_plus(ff_plus(pa, ff_neg(th)), ff_neg(Sm.y))};
  fc J0p, J1p, J0m, J1m;
  ff_j01(Pp, Ep, Bp, J0p, J1p);
  ff_j01(Pm, Em, Bm, J0m, J1m);
  const ff i2pi{0.15915493667125701904296875f, 6.4206382432985265e-09f};
  const ff w = ff_mult(i2pi, inv);
  // J_1 / s+- times s2: J_1p (Y + iX), J_1m (Y - iX)
  const ff tpx = ff_plus(ff_times(J1p.x, Y), ff_neg(ff_times(J1p.y, X)));
  const ff tpy = ff_plus(ff_times(J1p.x, X), ff_times(J1p.y, Y));
  const ff tmx = ff_plus(ff_times(J1m.x, Y), ff_times(J1m.y, X));
  const ff tmy = ff_plus(ff_times(J1m.y, Y), ff_neg(ff_times(J1m.x, X)));
  v[0] = ff_mult(i2pi, ff_plus(half_ln, ff_plus(J0p.x, J0m.x))).h;
  v[1] = ff_mult(i2pi, ff_plus(J0p.y, J0m.y)).h;
  v[2] = ff_mult(w, ff_plus(ff{X, 0.0f}, ff_plus(tmy, ff_neg(tpy)))).h;
  v[3] = ff_mult(w, ff_plus(tpx, ff_neg(tmx))).h;
  v[4] = ff_mult(w, ff_plus(ff{Y, 0.0f}, ff_neg(ff_plus(tpx, tmx)))).h;
  v[5] = -ff_mult(w, ff_plus(tpy, tmy)).h;
}
