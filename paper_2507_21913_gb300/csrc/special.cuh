// special.cuh -- device evaluation of the integrals I_n of Eq. generalintegral.
//
// With s = y - i x and P = kappa s (the substitution t = lambda s of Lemma 3.2
// and Appendix A),
//     I_n(x, y) = J_n(P) / (2 pi n! s^n),
//     J_n(P)    = int_S t^n e^{-t} / (t - P) dt,
// where S is the ray through s and, for real kappa, the path passes below the
// pole (Eq. dzGreensfunimplossless).  J_n satisfies the recursion of
// Eq. integralrecursion in the form J_n = (n-1)! + P J_{n-1}.
//
// Closed forms used (derived from the contour rotation of Appendix A):
//   J_0(P) = e^{-P} [ i pi - Ei(P) ],  Ei(P) = gamma + Log P + sum_{k>=1} P^k/(k k!)
// with the principal Log (arg P lies in (-pi/2, pi) for Re kappa > 0,
// Im kappa >= 0, y > 0), and for n >= 1 the same function continued term by term:
//   J_n(P) = e^{-P} [ P^n (i pi - Log P + psi(n+1)) - n! sum_{k != n} P^k / ((k-n) k!) ]
// (the exponential-integral series, A&S 5.1.12, with E_{n+1}(-P) and the residue
// term combined).  These power series are used where they do not cancel:
// |P| <= 1/2 or |P| - Re P <= 3/2 (P near the positive real axis; the
// cancellation factor is at most e^{|P| - Re P}).  Elsewhere the continued
// fraction of A&S 5.1.22 for e^{z} E_{n+1}(z) at z = -P (modified Lentz
// algorithm) gives K_n = n! e^{-P} E_{n+1}(-P), and
//   J_n = K_n + 2 pi i H P^n e^{-P},  H = 1 (Im P < 0), 1/2 (Im P = 0), 0 (Im P > 0),
// the residue rule of Appendix A.  J_n for all n <= K is obtained from J_{n*},
// n* = min(K, floor |P|), by the recursion run downwards (stable for n <= |P|)
// and upwards (stable for n >= |P|); the forward recursion from J_0 alone
// loses about |P|/2.3 digits (Lemma 3.2's regime n >= e|P| is where it is
// safe).  Supported range: |P| <= 60 (relative error ~1e-13 or better).
#pragma once
#include <mutex>

#include "common.cuh"
#include "mirror_ff.cuh"

#define HP_EULER_GAMMA 0.57721566490153286061
#define HP_PI 3.14159265358979323846
#define HP_TWO_PI 6.28318530717958647692

// reciprocals 1/k, k = 0..kRecip-1 (entry 0 unused).  Each translation unit
// that includes this header has its own copy (no relocatable device code);
// special_init_here() fills it once per device.
constexpr int kRecip = 512;
static __constant__ double c_recip[kRecip];
// Coefficients of the J_0 and J_1 power series (j01_arg), c_ser[0][k] = 1/(k k!)
// and c_ser[1][k] = 1/((k-1) k!), and the terms they need: c_nser[i] for
// |P| <= (i + 1) / 4 (a^N / N! <= 1e-18, well below the rounding of the sum).
constexpr int kSer = 64, kNser = 16;
static __constant__ double c_ser[2][kSer];
static __constant__ int c_nser[kNser];
static inline hpfmm_status special_init_here() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    set_last_error("special_init: no current device");
    return HPFMM_ECUDA;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return HPFMM_OK;
  static double host[kRecip];
  host[0] = 0.0;
  for (int k = 1; k < kRecip; ++k) host[k] = 1.0 / (double)k;
  HP_CUDA(cudaMemcpyToSymbol(c_recip, host, sizeof host));
  static double ser[2][kSer];
  static int nser[kNser];
  double f = 1.0;  // k!
  for (int k = 0; k < kSer; ++k) {
    if (k > 1) f *= (double)k;
    ser[0][k] = k > 0 ? 1.0 / ((double)k * f) : 0.0;
    ser[1][k] = k > 1 ? 1.0 / ((double)(k - 1) * f) : 0.0;
  }
  for (int i = 0; i < kNser; ++i) {
    const double a = 0.25 * (i + 1);
    double t = 1.0;
    int k = 0;
    while (k < kSer - 1 && (k < a || t > 1e-18)) t *= a / (double)++k;
    nser[i] = k;
  }
  HP_CUDA(cudaMemcpyToSymbol(c_ser, ser, sizeof ser));
  HP_CUDA(cudaMemcpyToSymbol(c_nser, nser, sizeof nser));
  done[dev] = true;
  return HPFMM_OK;
}
__device__ __forceinline__ double recip_int(int k) {  // 1/k for 0 < |k| < kRecip
  return k > 0 ? c_recip[k] : -c_recip[-k];
}

__device__ __forceinline__ bool jn_use_series(cd P) {
  double a = sqrt(abs2(P));
  return a <= 0.5 || (a - P.x) <= 1.5;
}

// J_n by the power series (valid for all P; used where it does not cancel)
__device__ inline cd jn_series(cd P, int n) {
  double a = sqrt(abs2(P));
  double psi = -HP_EULER_GAMMA;
  double nfact = 1.0;
  for (int k = 1; k <= n; ++k) {
    psi += c_recip[k];
    nfact *= k;
  }
  cd term = mk(1.0, 0.0);  // P^k / k!
  cd tot = mk(0.0, 0.0);
  cd Pn = mk(1.0, 0.0);
  for (int k = 0; k < kRecip - 1 && k - n < kRecip; ++k) {
    if (k == n) {
      Pn = term;  // P^n / n!
    } else {
      const double inv = recip_int(k - n);
      cd c = inv * term;
      tot = tot + c;
      if (k > n && k > a && abs2(c) < 1e-34 * abs2(tot)) break;
    }
    term = c_recip[k + 1] * (term * P);
  }
  // P^n (i pi - Log P + psi) - n! tot = n! [ (P^n/n!)(i pi - Log P + psi) - tot ]
  cd L = clog_d(P);
  cd br = mk(psi - L.x, HP_PI - L.y);
  cd v = nfact * (Pn * br - tot);
  return cexp_d(-P) * v;
}

// J_n by the continued fraction for E_{n+1} plus the residue rule
__device__ inline cd jn_cf(cd P, int n) {
  const double tiny = 1e-300;
  cd z = -P;
  double m = n + 1;
  // e^{z} E_m(z) = 1 / (z + m - 1*m / (z + m + 2 - 2(m+1) / (z + m + 4 - ...)))
  cd b = mk(z.x + m, z.y);
  cd f = (abs2(b) == 0) ? mk(tiny, 0.0) : b;
  cd C = f, D = mk(0.0, 0.0);
  for (int k = 1; k < 400; ++k) {
    double ak = -(double)k * (m + k - 1);
    b = mk(z.x + m + 2.0 * k, z.y);
    D = b + ak * D;
    if (abs2(D) == 0) D = mk(tiny, 0.0);
    D = cinv(D);
    C = b + ak * cinv(C);
    if (abs2(C) == 0) C = mk(tiny, 0.0);
    cd delta = C * D;
    f = f * delta;
    if (fabs(delta.x - 1.0) + fabs(delta.y) < 1e-16) break;
  }
  double nfact = 1.0;
  for (int k = 2; k <= n; ++k) nfact *= k;
  cd K = nfact * cinv(f);
  double H = (P.y < 0) ? 1.0 : ((P.y == 0) ? 0.5 : 0.0);
  if (H != 0.0) {
    cd Pn = mk(1.0, 0.0);
    for (int k = 0; k < n; ++k) Pn = Pn * P;
    cd r = (HP_TWO_PI * H) * mul_i(Pn * cexp_d(-P));
    K = K + r;
  }
  return K;
}

__device__ inline cd jn_direct(cd P, int n) {
  return jn_use_series(P) ? jn_series(P, n) : jn_cf(P, n);
}

// Values needed in single precision only: the series also where cancellation
// costs it up to a factor e^{|P| - Re P} <= e^10 of its double precision
// (relative error below 1e-10 for n <= 80, |P| <= 30, measured against
// 40-digit values of n! e^{-P} E_{n+1}(-P) plus the residue term).  There it
// takes 30 to 100 steps of one complex product, where the continued fraction
// takes up to 150 iterations of four divisions.
__device__ inline cd jn_direct_single(cd P, int n) {
  const double a = sqrt(abs2(P));
  const bool series = jn_use_series(P) || (a - P.x <= 10.0 && a <= 30.0);
  return series ? jn_series(P, n) : jn_cf(P, n);
}

// kappa with its logarithm ln|kappa| + i arg kappa, computed once on the host
struct KappaLog {
  cd kappa;
  double lk, ak;
  KappaFF f;  // the same in float pairs
};
inline KappaLog kappa_log(double kre, double kim) {
  KappaLog K;
  K.kappa = mk(kre, kim);
  K.lk = 0.5 * log(kre * kre + kim * kim);
  K.ak = atan2(kim, kre);
  K.f = KappaFF{ff_of(kre), ff_of(kim), ff_of(K.lk), ff_of(K.ak), kim == 0.0};
  return K;
}

// sum_{k=0}^{N-1} c[k] z^k for real coefficients and complex z by the real
// recurrence b_k = c_k + 2 Re(z) b_{k+1} - |z|^2 b_{k+2} (the quotient of the
// polynomial by z^2 - 2 Re(z) z + |z|^2): two FP64 instructions a term, where
// Horner's rule in complex arithmetic takes four.
template <int N>
__device__ __forceinline__ cd real_poly(const double (&c)[N], cd z, double z2) {
  double b1 = c[N - 1], b2 = 0.0;
  const double r = z.x + z.x;
#pragma unroll
  for (int k = N - 2; k >= 1; --k) {
    const double t = fma(r, b1, fma(-z2, b2, c[k]));
    b2 = b1;
    b1 = t;
  }
  return mk(fma(z.x, b1, fma(-z2, b2, c[0])), z.y * b1);
}

// e^{-P} and sum_{k>=1} P^k/(k k!) to P^N, P2 = |P|^2 (N <= 10)
template <int N>
__device__ __forceinline__ void exp_sum_poly(cd P, double P2, cd &E, cd &S) {
  const double ce[11] = {1.0, 1.0, 1.0 / 2.0, 1.0 / 6.0, 1.0 / 24.0, 1.0 / 120.0, 1.0 / 720.0,
                         1.0 / 5040.0, 1.0 / 40320.0, 1.0 / 362880.0, 1.0 / 3628800.0};
  const double cs[11] = {0.0, 1.0, 1.0 / 4.0, 1.0 / 18.0, 1.0 / 96.0, 1.0 / 600.0,
                         1.0 / 4320.0, 1.0 / 35280.0, 1.0 / 322560.0, 1.0 / 3265920.0,
                         1.0 / 36288000.0};
  double e[N], s[N];
#pragma unroll
  for (int k = 0; k < N; ++k) {
    e[k] = ce[k + 1];
    s[k] = cs[k + 1];
  }
  const cd mP = mk(-P.x, -P.y);
  E = mP * real_poly<N>(e, mP, P2);
  E.x += 1.0;
  S = P * real_poly<N>(s, P, P2);
}

// J_0 and J_1 of one argument, |P| = a, given Log P = lr + i arg and e^{-P}: the
// power series where it does not cancel (the region of jn_use_series), J_0
// below |P| = 1 and J_1 above (where 1 + P J_0 would cancel), each with
// J_1 = 1 + P J_0 for the other; the general forms elsewhere (beyond |P| = 4 the
// recurrence of real_poly would lose about |P| of the series' precision).
__device__ __forceinline__ void j01_arg(cd P, double P2, float a, double lr, double arg, cd E,
                                        cd &J0, cd &J1) {
  const bool big = P2 >= 1.0;
  if (a <= 0.5f || (a <= 4.0f && (double)a - P.x <= 1.5)) {
    // each lane its own term count, so that a pair's value does not depend on the
    // pairs beside it
    const int N = c_nser[min((int)(4.0f * a), kNser - 1)];
    const double r = P.x + P.x;
    double b1 = 0.0, b2 = 0.0;
    if (!big) {
      for (int k = N; k >= 2; --k) {
        const double t = fma(r, b1, fma(-P2, b2, c_ser[0][k]));
        b2 = b1;
        b1 = t;
      }
      // sum_{k>=1} c_k P^(k-1)
      const cd S = P * mk(fma(P.x, b1, fma(-P2, b2, 1.0)), P.y * b1);
      J0 = E * mk(-HP_EULER_GAMMA - lr - S.x, HP_PI - arg - S.y);
      const cd v = P * J0;
      J1 = mk(1.0 + v.x, v.y);
      return;
    }
    for (int k = N; k >= 3; --k) {
      const double t = fma(r, b1, fma(-P2, b2, c_ser[1][k]));
      b2 = b1;
      b1 = t;
    }
    // P sum_{k>=2} c_k P^(k-2), c_2 = 1/2, and the log terms
    const cd T = P * mk(fma(P.x, b1, fma(-P2, b2, 0.5)), P.y * b1);
    cd v = P * mk(1.0 - HP_EULER_GAMMA - lr - T.x, HP_PI - arg - T.y);
    v.x += 1.0;
    J1 = E * v;
  } else if (!big) {
    J0 = jn_cf(P, 0);
    const cd v = P * J0;
    J1 = mk(1.0 + v.x, v.y);
    return;
  } else {
    J1 = jn_direct(P, 1);
  }
  const double inv = 1.0 / P2;
  J0 = inv * (mk(P.x, -P.y) * mk(J1.x - 1.0, J1.y));
}

// J_0 and J_1 of both reaction arguments of one pair, P+ = kappa (Y - iX) and
// P- = kappa (Y + iX) (Y > 0), double precision, s2 = X^2 + Y^2 and its log
// given (the image term of the pair needs both).  Log P+- = Log kappa + ln|s|
// -+ i atan2(X, Y) (s+- = Y -+ iX are conjugate, and the sum of the arguments
// stays in (-pi/2, pi)), so one log and one atan2 serve both.  For |P| <= 1/8
// fixed-length series: 6 terms for |P| <= 1/64, 10 above (dropped terms below
// 1e-16 relative).  Beyond, j01_arg.  For real kappa the two arguments are
// conjugate and J_n(conj P) = conj J_n(P) + 2 pi i conj(P)^n e^{-conj P}
// (only the i pi of the seed is not conjugated): one evaluation, at the
// argument with Im P >= 0, whose value holds no residue term to cancel.
// FP64 instructions a pair, beside log and atan2: about 60 for |P| <= 1/8
// with real kappa, 200 for |P| about 1 (the series of each argument by complex
// Horner steps and a term-by-term test took about 250 and 1500).
__device__ __forceinline__ void j01_pm(const KappaLog &K, double X, double Y, double s2,
                                       double ln_s2, cd &J0p, cd &J1p, cd &J0m, cd &J1m) {
  const cd Pp = K.kappa * mk(Y, -X), Pm = K.kappa * mk(Y, X);
  const double a2 = abs2(K.kappa) * s2;
  const double lr = fma(0.5, ln_s2, K.lk), th = atan2(X, Y);
  const bool real = K.kappa.y == 0.0;
  if (a2 <= 1.0 / 64.0) {
    cd Ep, Sp, Em, Sm;
    if (a2 <= 1.0 / 4096.0) {
      exp_sum_poly<6>(Pp, a2, Ep, Sp);
      if (!real) exp_sum_poly<6>(Pm, a2, Em, Sm);
    } else {
      exp_sum_poly<10>(Pp, a2, Ep, Sp);
      if (!real) exp_sum_poly<10>(Pm, a2, Em, Sm);
    }
    if (real) {
      Em = conj(Ep);
      Sm = conj(Sp);
    }
    J0p = Ep * mk(-HP_EULER_GAMMA - lr - Sp.x, HP_PI - (K.ak - th) - Sp.y);
    J0m = Em * mk(-HP_EULER_GAMMA - lr - Sm.x, HP_PI - (K.ak + th) - Sm.y);
    const cd vp = Pp * J0p, vm = Pm * J0m;
    J1p = mk(1.0 + vp.x, vp.y);
    J1m = mk(1.0 + vm.x, vm.y);
    return;
  }
  const float a = sqrtf((float)a2);
  if (real) {
    const bool up = X > 0.0;  // P- has Im >= 0
    const cd P = up ? Pm : mk(Pp.x, Pp.y);
    const cd E = cexp_d(-P), Ec = conj(E);
    cd J0, J1;
    j01_arg(P, a2, a, lr, fabs(th), E, J0, J1);
    const cd r0 = HP_TWO_PI * mul_i(Ec), r1 = conj(P) * r0;
    const cd Q0 = conj(J0) + r0, Q1 = conj(J1) + r1;
    J0m = up ? J0 : Q0;
    J1m = up ? J1 : Q1;
    J0p = up ? Q0 : J0;
    J1p = up ? Q1 : J1;
  } else {
    j01_arg(Pp, a2, a, lr, K.ak - th, cexp_d(-Pp), J0p, J1p);
    j01_arg(Pm, a2, a, lr, K.ak + th, cexp_d(-Pm), J0m, J1m);
  }
}

// Single-precision J_0, J_1 for |P| <= 1 (near-field pairs of the fast path):
// J_0 = e^{-P}[i pi - gamma - Log P - sum_{k>=1} P^k/(k k!)], 11 terms.
__device__ __forceinline__ void j01_f(cf P, cf &J0, cf &J1) {
  cf term = P;
  cf s = P;
#pragma unroll
  for (int k = 2; k <= 11; ++k) {
    term = (1.0f / k) * (term * P);
    s = s + (1.0f / k) * term;
  }
  float lr = 0.5f * __logf(P.x * P.x + P.y * P.y);
  float th = atan2f(P.y, P.x);
  cf br = mk(-(float)HP_EULER_GAMMA - lr - s.x, (float)HP_PI - th - s.y);
  float e = __expf(-P.x), sn, cs;
  __sincosf(-P.y, &sn, &cs);
  cf eP = mk(e * cs, e * sn);
  J0 = eP * br;
  cf v = P * J0;
  J1 = mk(1.0f + v.x, v.y);
}
