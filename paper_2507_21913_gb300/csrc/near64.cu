// near64.cu -- near field of the double-precision plans on the uniform tree:
// the free-space pairs of the 3 x 3 leaf neighbourhood (Eq. 1.2) and, for the
// bottom leaf row, the image and reaction pairs (Eqs. reactioncomp1,
// reactioncomp2).  Both need only the sorted points and charges, so they run
// beside the far-field passes; the L2P kernel adds their sums.
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "ff64.cuh"
#include "pairs.cuh"
#include "special.cuh"

namespace {

// ln table of ff_log, filled once per device
__device__ ff g_log_tab[kFfLogN];

// exponent of the power of two above the leaf side: the unit of the
// fixed-point coordinates is 2^(kd - 60), so that differences between
// neighbouring leaves stay below 2^61, and ff_from_fixed's results are in
// units of 2^(kd - 23)
__device__ __forceinline__ int leaf_exponent(const DevGeom *dg, int H) {
  return (int)((__double_as_longlong(dg->side) >> 52) & 0x7ff) - 1022 - H;
}

// fixed-point coordinates and split charges of every point, in tree order.
// The charges are scaled by the power of two of the largest (qexp, its biased
// exponent, from the gather), so that their floats cannot leave the range.
__global__ void __launch_bounds__(256)
k_prep64(const double *__restrict__ xs, const double *__restrict__ ys,
         const double *__restrict__ qs, int64_t n, int H, const DevGeom *__restrict__ dg,
         const int *__restrict__ qexp, longlong2 *__restrict__ fxy, float2 *__restrict__ fq) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int s = 60 - leaf_exponent(dg, H);
  fxy[k] = make_longlong2(ff_fixed(xs[k], s), ff_fixed(ys[k], s));
  const ff q = ff_split_scaled(qs[k], *qexp - 1023);
  fq[k] = make_float2(q.h, q.l);
}

// The source ranges of a target's 3 x 3 neighbourhood, walked by a group of S
// lanes: lane g takes the entries g, g + S, ... of the ranges' concatenation.
struct NearWalk {
  int ix, iy, nx, r, k, end;
  const int *leaf_start;
  __device__ __forceinline__ void range(int rr, int &b, int &e) const {
    const int mx = ix + rr % 3 - 1, my = iy + rr / 3 - 1;
    b = e = 0;
    if (mx >= 0 && my >= 0 && mx < nx && my < nx) {
      const uint64_t m = box_morton(mx, my);
      b = leaf_start[m];
      e = leaf_start[m + 1];
    }
  }
  // to the range that holds the current entry
  __device__ __forceinline__ void settle() {
    while (k >= end && r < 8) {
      const int over = k - end;
      int b;
      range(++r, b, end);
      k = b + over;
    }
  }
  __device__ __forceinline__ void start(const int *ls, int leaf_ix, int leaf_iy, int n, int g) {
    leaf_start = ls;
    ix = leaf_ix;
    iy = leaf_iy;
    nx = n;
    r = -1;
    k = g;
    end = 0;
    settle();
  }
  __device__ __forceinline__ bool more() const { return k < end; }
  __device__ __forceinline__ void step(int S) {
    k += S;
    if (k >= end) settle();
  }
};

// Free-space pairs, S lanes a target (S a power of two, consecutive lanes).
// Sums to near[c n + i], c = 0..2: sum q ln r^2, sum q dx / r^2, sum q dy / r^2
// (the coincident and the target's own point as in pair_free: only j = i is
// left out).
//
// Bound by the single-precision issue slots: about 200 a pair (ff64.cuh), where
// the FP64 expression took about 47 FP64 instructions = 3600 slots: a step of
// 1e6 points at order 12 went from 28.4 to 4.65 ms (with the L2P taken out of
// the leaf kernel and the far field beside it).  The lanes
// of a warp are consecutive targets of two or three leaves; each walks its own
// neighbourhood, so none idles for another's leaf, and the loads of one leaf's
// lanes coincide.
//
// FF false: the pairs in FP64, for orders whose truncation error lies below the
// pairs' 2^-48 and for trees of one level, whose sum is near field only; the
// same where a charge is not finite (qexp at its top).
template <bool FF>
__global__ void __launch_bounds__(128)
k_near64(const double *__restrict__ xs, const double *__restrict__ ys,
         const double *__restrict__ qs, const longlong2 *__restrict__ fxy,
         const float2 *__restrict__ fq, const uint64_t *__restrict__ keys,
         const int *__restrict__ leaf_start, int64_t n, int H, int S,
         const DevGeom *__restrict__ dg, const int *__restrict__ qexp,
         double *__restrict__ near) {
  __shared__ ff tab[kFfLogN];
  const int qe = FF ? *qexp : 0;
  const bool fast = FF && qe != 0x7ff;
  if (fast) {
    for (int e = threadIdx.x; e < kFfLogN; e += blockDim.x) tab[e] = g_log_tab[e];
    __syncthreads();
  }
  const int g = (int)(threadIdx.x & (S - 1)), per = (int)blockDim.x / S;
  for (int64_t t0 = (int64_t)blockIdx.x * per; t0 < n; t0 += (int64_t)gridDim.x * per) {
    const int64_t ti = t0 + (int)threadIdx.x / S;
    const bool act = ti < n;
    const int i = act ? (int)ti : 0;
    double lf = 0.0, gx = 0.0, gy = 0.0;
    if (act) {
      const uint64_t leaf = keys[i] >> (60 - 2 * H);
      NearWalk w;
      w.start(leaf_start, box_ix(leaf), box_iy(leaf), 1 << H, g);
      if (fast) {
        // r^2 in units of 2^(2 kd - 46): the exponent's part of the log
        const int ebias = 46 - 2 * leaf_exponent(dg, H);
        const longlong2 me = fxy[i];
        ff_sum3 sl{0.f, 0.f, 0.f}, sk{0.f, 0.f, 0.f}, sx{0.f, 0.f, 0.f}, sy{0.f, 0.f, 0.f};
        for (; w.more(); w.step(S)) {
          const longlong2 s = fxy[w.k];
          const float2 qv = fq[w.k];
          const int64_t DX = me.x - s.x, DY = me.y - s.y;
          const int hx = (int)(DX >> 32), hy = (int)(DY >> 32);
          if (((hx ^ (hx >> 31)) | (hy ^ (hy >> 31))) == 0) {
            // closer than 2^-28 of the leaf side, where the fixed-point unit
            // could show, or the target itself
            if (w.k != i) {
              const double dx = xs[i] - xs[w.k], dy = ys[i] - ys[w.k];
              PairAcc<double> a;
              pair_free(a, dx, dy, qs[w.k]);
              lf += a.lf;
              gx += a.gfx;
              gy += a.gfy;
            }
            continue;
          }
          const ff dx = ff_from_fixed(DX), dy = ff_from_fixed(DY), q{qv.x, qv.y};
          const ff r2 = ff_norm2(dx, dy);
          const float c = ff_rcp_approx(r2.h);
          float k;
          sl.add(ff_prod(ff_log(r2, c, tab, ebias, k), q));
          sk.add(ff_prod(ff{k, 0.f}, q));
          const ff qw = ff_prod(ff_recip(r2, c), q);
          sx.add(ff_prod(qw, dx));
          sy.add(ff_prod(qw, dy));
        }
        const double us = ldexp(1.0, qe - 1023);
        const double ug = ldexp(1.0, qe - 1023 + 23 - leaf_exponent(dg, H));
        lf += us * fma(0.69314718055994530942, sk.value(), sl.value());
        gx += ug * sx.value();
        gy += ug * sy.value();
      } else {
        PairAcc<double> a;
        const double x = xs[i], y = ys[i];
        for (; w.more(); w.step(S))
          if (w.k != i) pair_free(a, x - xs[w.k], y - ys[w.k], qs[w.k]);
        lf = a.lf;
        gx = a.gfx;
        gy = a.gfy;
      }
    }
    for (int o = S >> 1; o > 0; o >>= 1) {
      lf += __shfl_xor_sync(0xffffffffu, lf, o);
      gx += __shfl_xor_sync(0xffffffffu, gx, o);
      gy += __shfl_xor_sync(0xffffffffu, gy, o);
    }
    if (act && g == 0) {
      near[i] = lf;
      near[n + i] = gx;
      near[2 * n + i] = gy;
    }
  }
}

// Image and reaction pairs of the bottom leaf row, assigned to the outputs
// (the L2P adds to them).  One warp a target, its lanes over the sources of the
// three bottom-row neighbours, then butterfly sums.  Bound by the FP64 pipe,
// about 250 instructions a pair: what counts is that the pairs of the few
// bottom-row targets spread over all SMs (2000 points at order 12, one lane a
// target: 8.1 ms a call; so: 0.74 ms).
constexpr int kMir64Warps = 4, kMir64Split = 16;
__global__ void __launch_bounds__(32 * kMir64Warps)
k_mirror64(const double *__restrict__ xs, const double *__restrict__ ys,
           const double *__restrict__ qs, const int64_t *__restrict__ perm,
           const int *__restrict__ leaf_start, int H, KappaLog K, double *__restrict__ pot,
           double *__restrict__ grad) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nx = 1 << H, ix = blockIdx.x;
  const uint64_t leaf = box_morton(ix, 0);
  const int b0 = leaf_start[leaf], b1 = leaf_start[leaf + 1];
  int s0[3], cnt[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const int mx = ix - 1 + k;
    s0[k] = cnt[k] = 0;
    if (mx >= 0 && mx < nx) {
      const uint64_t sl = box_morton(mx, 0);
      s0[k] = leaf_start[sl];
      cnt[k] = leaf_start[sl + 1] - s0[k];
    }
  }
  const int ns = cnt[0] + cnt[1] + cnt[2];
  const int stride = kMir64Warps * (int)gridDim.y;
  for (int i = b0 + warp + kMir64Warps * (int)blockIdx.y; i < b1; i += stride) {
    const double x = xs[i], y = ys[i];
    PairAcc<double> a;
    for (int r = lane; r < ns; r += 32) {
      const int j = r < cnt[0] ? s0[0] + r
                               : (r < cnt[0] + cnt[1] ? s0[1] + r - cnt[0]
                                                      : s0[2] + r - cnt[0] - cnt[1]);
      pair_mirror_d(a, x - xs[j], y + ys[j], qs[j], K);
    }
    double v[9] = {a.li, a.gix, a.giy, a.ur.x, a.ur.y, a.grx.x, a.grx.y, a.gry.x, a.gry.y};
#pragma unroll
    for (int e = 0; e < 9; ++e)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v[e] += __shfl_xor_sync(0xffffffffu, v[e], o);
    if (lane == 0) {
      PairAcc<double> s;
      s.li = v[0];
      s.gix = v[1];
      s.giy = v[2];
      s.ur = mk(v[3], v[4]);
      s.grx = mk(v[5], v[6]);
      s.gry = mk(v[7], v[8]);
      cd u, gx, gy;
      s.finish(u, gx, gy);
      const int64_t o = perm[i];
      pot[2 * o] = u.x;
      pot[2 * o + 1] = u.y;
      if (grad) {
        grad[4 * o + 0] = gx.x;
        grad[4 * o + 1] = gx.y;
        grad[4 * o + 2] = gy.x;
        grad[4 * o + 3] = gy.y;
      }
    }
  }
}

}  // namespace

hpfmm_status near64_prepare() {
  static std::mutex mu;
  static bool done[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();
    set_last_error("near64_prepare: no current device");
    return HPFMM_ECUDA;
  }
  std::lock_guard<std::mutex> lock(mu);
  if (done[dev]) return special_init_here();
  static ff tab[kFfLogN];
  ff_log_table(tab);
  HP_CUDA(cudaMemcpyToSymbol(g_log_tab, tab, sizeof tab));
  HP_CUDA(prefer_shared(k_prep64));
  HP_CUDA(prefer_shared(k_near64<true>));
  HP_CUDA(prefer_shared(k_near64<false>));
  HP_CUDA(prefer_shared(k_mirror64));
  done[dev] = true;
  return special_init_here();
}

namespace {
// The pairs' 2^-48 adds about 1e-15 to the relative error of the potential and
// 4e-15 to the gradient's.  Up to order 28 that is below a tenth of the far
// field's truncation (about 1.5e-14 and 6e-13 at 28, measured for 1000 to 60000
// points); higher orders, and trees of one level, which have no free far
// field, take FP64 pairs.
bool near64_fast(const hpfmm_plan *pl) { return pl->p <= 28 && pl->H >= 2; }
}  // namespace

// Blocks per SM of the float-pair kernel, which loops over the targets: the far
// field's kernels, bound by the FP64 pipe with few warps, find room beside them.
constexpr int kNearBlocks = 5;

int near64_kernels(const hpfmm_plan *pl) { return near64_fast(pl) ? 2 : 1; }

// The lanes per target: enough threads to fill the chip (measured at 2000 and
// 40009 points), one lane a target from 131072 points on.
hpfmm_status near64_launch(hpfmm_plan *pl, const double *qs, cudaStream_t st) {
  const int64_t n = pl->n;
  int S = 1;
  while (S < 32 && n * S < (1 << 17)) S <<= 1;
  const unsigned nb = (unsigned)((n * S + 127) / 128);
  if (near64_fast(pl)) {
    k_prep64<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(pl->xs, pl->ys, qs, n, pl->H, pl->dgeom,
                                                          pl->qexp, (longlong2 *)pl->fxy,
                                                          (float2 *)pl->fq);
    const unsigned most = (unsigned)(kNearBlocks * pl->sms);
    k_near64<true><<<nb < most ? nb : most, 128, 0, st>>>(pl->xs, pl->ys, qs, (const longlong2 *)pl->fxy,
                                       (const float2 *)pl->fq, pl->keys, pl->leaf_start, n, pl->H,
                                       S, pl->dgeom, pl->qexp, pl->near64);
  } else {
    k_near64<false><<<nb, 128, 0, st>>>(pl->xs, pl->ys, qs, nullptr, nullptr, pl->keys,
                                        pl->leaf_start, n, pl->H, S, pl->dgeom, pl->qexp,
                                        pl->near64);
  }
  HP_LAUNCH_CHECK();
  return HPFMM_OK;
}

hpfmm_status mirror64_launch(hpfmm_plan *pl, const double *qs, double *pot, double *grad,
                             cudaStream_t st) {
  k_mirror64<<<dim3((unsigned)(1 << pl->H), kMir64Split), 32 * kMir64Warps, 0, st>>>(
      pl->xs, pl->ys, qs, pl->perm, pl->leaf_start, pl->H, kappa_log(pl->kre, pl->kim), pot, grad);
  HP_LAUNCH_CHECK();
  return HPFMM_OK;
}
