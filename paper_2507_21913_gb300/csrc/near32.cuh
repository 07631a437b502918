// near32.cuh -- single-precision near-field helpers shared by the uniform
// and the adaptive leaf kernels: SFU reciprocal and log2, an integer
// float -> double conversion, and the image + reaction pair of two points of
// the bottom leaf row (Eqs. reactioncomp1, reactioncomp2).
#pragma once
#include <mutex>

#include "common.cuh"
#include "special.cuh"

__device__ __forceinline__ float fast_rcp(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float fast_lg2(float x) {
  float r;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// float -> double by re-biasing the exponent with integer operations (the
// FP64 conversion instruction runs on GB300's narrow FP64 pipe); denormal
// single-precision inputs become 0, infinities and NaNs are kept
__device__ __forceinline__ double f2d(float v) {
  const unsigned u = __float_as_uint(v);
  const unsigned e = (u >> 23) & 0xffu;
  unsigned long long r = (unsigned long long)(u & 0x80000000u) << 32;
  if (e == 0xffu) r |= (0x7ffull << 52) | ((unsigned long long)(u & 0x7fffffu) << 29);
  else if (e != 0) r |= ((unsigned long long)(e + 896u) << 52) | ((unsigned long long)(u & 0x7fffffu) << 29);
  return __longlong_as_double((long long)r);
}

// single-precision sums of one target's free-space pairs
struct NearAcc {
  float lf, gx, gy;  // sum q log2 r^2, sum q (dx, dy) / r^2
};

// The image and reaction pair of two points of the bottom leaf row for a unit
// charge: u and its gradient, with the 1/2pi and 1/4pi factors.  They do not
// depend on the charge, so many charge vectors share one evaluation.
struct MirrorVal {
  float ur, ui, gxr, gxi, gyr, gyi;
};

// in double precision, rounded: out of line, as the single-precision kernels
// need it for few pairs
static __device__ __noinline__ MirrorVal mirror_value_d(const KappaLog &K, double X, double Y) {
  const double s2 = X * X + Y * Y, ln = log(s2), inv = 1.0 / s2;
  cd J0p, J1p, J0m, J1m;
  j01_pm(K, X, Y, s2, ln, J0p, J1p, J0m, J1m);
  const double i2pi = 1.0 / HP_TWO_PI, w = i2pi * inv;
  const cd tp = J1p * mk(Y, X), tm = J1m * mk(Y, -X);  // J_1 / s+- times s2
  MirrorVal v;
  v.ur = (float)(i2pi * (0.5 * ln + J0p.x + J0m.x));
  v.ui = (float)(i2pi * (J0p.y + J0m.y));
  v.gxr = (float)(w * (X - (tp.y - tm.y)));
  v.gxi = (float)(w * (tp.x - tm.x));
  v.gyr = (float)(w * (Y - (tp.x + tm.x)));
  v.gyi = (float)(-w * (tp.y + tm.y));
  return v;
}

// tables of the float-pair form (mirror_ff.cuh), one copy per translation unit
// that includes this header; mirror_tables_here() fills them once per device
static __device__ ff g_mir_log[kFfLogN];
static __device__ FfAngle g_mir_angle[kFfAng];
static inline hpfmm_status mirror_tables_here() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    set_last_error("mirror_tables: no current device");
    return HPFMM_ECUDA;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return HPFMM_OK;
  static ff lt[kFfLogN];
  static FfAngle at[kFfAng];
  ff_log_table(lt);
  ff_angle_table(at);
  HP_CUDA(cudaMemcpyToSymbol(g_mir_log, lt, sizeof lt));
  HP_CUDA(cudaMemcpyToSymbol(g_mir_angle, at, sizeof at));
  done[dev] = true;
  return HPFMM_OK;
}

// in float pairs, rounded (out of line as well)
static __device__ __noinline__ MirrorVal mirror_value_ff(const KappaLog &K, float X, float Y) {
  float v[6];
  ff_mirror(X, Y, K.f, atan2f(fabsf(X), Y), g_mir_log, g_mir_angle, v);
  return MirrorVal{v[0], v[1], v[2], v[3], v[4], v[5]};
}

// kappa as the single-precision pair uses it
struct KappaF {
  cf kappa;
  float a2, lk, ak;  // |kappa|^2, ln |kappa|, arg kappa
  bool real;
};
__device__ __forceinline__ KappaF kappa_f(const KappaLog &K) {
  return KappaF{mk((float)K.kappa.x, (float)K.kappa.y), (float)abs2(K.kappa), (float)K.lk,
                (float)K.ak, K.kappa.y == 0.0};
}

// e^{-P} and sum_{k=1}^{11} P^k/(k k!) in single precision, P2 = |P|^2 <= 1, by
// the real recurrence of real_poly
__device__ __forceinline__ void exp_sum_f(cf P, float P2, cf &E, cf &S) {
  const float c[11] = {1.0f,           1.0f / 4.0f,      1.0f / 18.0f,     1.0f / 96.0f,
                       1.0f / 600.0f,  1.0f / 4320.0f,   1.0f / 35280.0f,  1.0f / 322560.0f,
                       1.0f / 3265920.0f, 1.0f / 36288000.0f, 1.0f / 439084800.0f};
  float b1 = c[10], b2 = 0.0f;
  const float r = P.x + P.x;
#pragma unroll
  for (int k = 9; k >= 1; --k) {
    const float t = fmaf(r, b1, fmaf(-P2, b2, c[k]));
    b2 = b1;
    b1 = t;
  }
  S = P * mk(fmaf(P.x, b1, fmaf(-P2, b2, c[0])), P.y * b1);
  const float e = __expf(-P.x);
  float sn, cs;
  __sincosf(-P.y, &sn, &cs);
  E = mk(e * cs, e * sn);
}

// Single precision where the series is accurate (|P| <= 1) and the pair is not
// below tau, else float pairs (|P| <= 1/8, s2 well inside the float range; 4e6
// clustered points in MIXED mode: 7.87 ms a step with FP64, 5.45 so) or double.  X
// the difference of the x, Y the sum of the y.  The reciprocal of X^2 + Y^2 serves the
// image and both reaction terms, and for real kappa the arguments P+- are conjugate,
// J_n(conj P) = conj J_n(P) + 2 pi i conj(P)^n e^{-conj P}: about 130 instructions a
// pair (two complex series, four divisions and the accumulation for one charge took
// about 450).
__device__ __forceinline__ MirrorVal mirror_value(float X, float Y, const KappaF &kf,
                                                  const KappaLog &K, float tau) {
  const float s2 = fmaf(X, X, Y * Y), P2 = kf.a2 * s2;
  if (!(P2 <= 1.0f && Y >= tau))
    return P2 <= 0.0156f && s2 >= 1e-24f ? mirror_value_ff(K, X, Y) : mirror_value_d(K, X, Y);
  const float ln = 0.693147180559945f * fast_lg2(s2), inv = fast_rcp(s2);
  // (ln |P| of its own: as ln |s| + ln |kappa| it loses what the two cancel; that for
  // P2 near the end of the float range)
  const float lr = P2 > 1e-30f ? 0.346573590279973f * fast_lg2(P2) : fmaf(0.5f, ln, kf.lk);
  const float th = atan2f(X, Y);
  const float g = -(float)HP_EULER_GAMMA - lr, pi = (float)HP_PI;
  const cf Pp = kf.kappa * mk(Y, -X), Pm = kf.kappa * mk(Y, X);
  cf Ep, Sp, Em, Sm;
  exp_sum_f(Pp, P2, Ep, Sp);
  if (kf.real) {
    Em = conj(Ep);
    Sm = conj(Sp);
  } else {
    exp_sum_f(Pm, P2, Em, Sm);
  }
  const cf J0p = Ep * mk(g - Sp.x, pi - (kf.ak - th) - Sp.y);
  const cf J0m = Em * mk(g - Sm.x, pi - (kf.ak + th) - Sm.y);
  cf J1p = Pp * J0p, J1m = Pm * J0m;
  J1p.x += 1.0f;
  J1m.x += 1.0f;
  const cf tp = J1p * mk(Y, X), tm = J1m * mk(Y, -X);
  const float i2pi = (float)(1.0 / HP_TWO_PI), w = i2pi * inv;
  MirrorVal v;
  v.ur = i2pi * (0.5f * ln + (J0p.x + J0m.x));
  v.ui = i2pi * (J0p.y + J0m.y);
  v.gxr = w * (X - (tp.y - tm.y));
  v.gxi = w * (tp.x - tm.x);
  v.gyr = w * (Y - (tp.x + tm.x));
  v.gyi = -w * (tp.y + tm.y);
  return v;
}

// sums over the sources of one target
struct MirrorAcc {
  float v[6];
  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int e = 0; e < 6; ++e) v[e] = 0.0f;
  }
  __device__ __forceinline__ void add(float q, const MirrorVal &m) {
    v[0] = fmaf(q, m.ur, v[0]);
    v[1] = fmaf(q, m.ui, v[1]);
    v[2] = fmaf(q, m.gxr, v[2]);
    v[3] = fmaf(q, m.gxi, v[3]);
    v[4] = fmaf(q, m.gyr, v[4]);
    v[5] = fmaf(q, m.gyi, v[5]);
  }
  // over the G lanes of an aligned group
  template <int G>
  __device__ __forceinline__ void reduce(unsigned mask) {
#pragma unroll
    for (int e = 0; e < 6; ++e)
#pragma unroll
      for (int o = G / 2; o > 0; o >>= 1) v[e] += __shfl_xor_sync(mask, v[e], o);
  }
  // to the outputs of point o: assigned, or added to what is there (a double at a
  // time: the caller's complex arrays need no more than a double's alignment)
  __device__ __forceinline__ void put(double *pot, double *grad, int64_t o, bool assign) const {
    double *po = pot + 2 * o, *go = grad + 4 * o;
    double a[6];
#pragma unroll
    for (int e = 0; e < 6; ++e) a[e] = f2d(v[e]);
    if (!assign) {
      a[0] += po[0];
      a[1] += po[1];
    }
    po[0] = a[0];
    po[1] = a[1];
    if (!grad) return;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (!assign) a[2 + e] += go[e];
      go[e] = a[2 + e];
    }
  }
};
