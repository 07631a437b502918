// near64.cu -- near field of the double-precision plans on the uniform tree:
// the free-space pairs of the 3 x 3 leaf neighbourhood (Eq. 1.2) and, for the
// bottom leaf row, the image and reaction pairs (Eqs. reactioncomp1,
// reactioncomp2).  Both need only the sorted points and charges, so they run
// beside the far-field passes; the L2P kernel adds their sums.
#include <math.h>

#include <mutex>

#include "common.cuh"
#include "fix64.cuh"
#include "pairs.cuh"
#include "special.cuh"

namespace {

// ln table of fx_pair, filled once per device
__device__ int64_t g_log_tab[kFfLogN];

// exponent of the power of two above the leaf side (fix64.cuh, kd)
__device__ __forceinline__ int leaf_exponent(const DevGeom *dg, int H) {
  return (int)((__double_as_longlong(dg->side) >> 52) & 0x7ff) - 1022 - H;
}

// a point's charge and the lowest 32 bits of its fixed-point coordinates, of
// which the charge's drop (fix64.cuh) takes the last five of x
struct __align__(16) FxRest {
  int64_t q;
  uint32_t ex, ey;
  __device__ __forceinline__ int drop() const { return (int)(ex & 31u); }
};

// fixed-point coordinates and charges of every point, in tree order
__global__ void __launch_bounds__(256)
k_prep64(const double *__restrict__ xs, const double *__restrict__ ys,
         const double *__restrict__ qs, int64_t n, int H, const DevGeom *__restrict__ dg,
         const int *__restrict__ qexp, ulonglong2 *__restrict__ fxy, FxRest *__restrict__ fq) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= n) return;
  const int s = 60 - leaf_exponent(dg, H);
  const fx96 x = fx_fixed(xs[k], s), y = fx_fixed(ys[k], s);
  const FxCharge q = fx_charge(qs[k], *qexp >> 1);
  fxy[k] = make_ulonglong2(x.v, y.v);
  fq[k] = FxRest{q.bits, (x.e & ~31u) | (uint32_t)q.drop, y.e};
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
// Bound by the integer pipes, adder and multiplier at half the issue rate each:
// about 215 warp instructions a pair with the walk, 100 of the one and 90 of the
// other (fix64.cuh).  A step of 1e6 points at order 12, far field beside it, takes
// 3.12 ms; 28.4 ms with FP64 pairs, 3.01 ms with pairs of floats, which held 48
// bits and lost digits next to the axes.  The lanes of a warp are consecutive
// targets of two or three leaves; each walks its own neighbourhood, so none idles
// for another's leaf, and the loads of one leaf's lanes coincide.
//
// FIX false: the pairs in FP64, for orders above 28 and for trees of one level,
// whose sum is near field only; the same in either form for pairs closer than
// fx_cut and where the largest charge is subnormal or not finite (qexp 1, or at
// its top).
template <bool FIX>
__global__ void __launch_bounds__(128, 8)
k_near64(const double *__restrict__ xs, const double *__restrict__ ys,
         const double *__restrict__ qs, const ulonglong2 *__restrict__ fxy,
         const FxRest *__restrict__ fq, const uint64_t *__restrict__ keys,
         const int *__restrict__ leaf_start, int64_t n, int H, int S,
         const DevGeom *__restrict__ dg, const int *__restrict__ qexp,
         double *__restrict__ near) {
  __shared__ int64_t tab[kFfLogN];
  const int qe = FIX ? *qexp : 0;
  const bool fast = FIX && qe != 1 && qe < 2 * 0x7ff;
  const int kd = leaf_exponent(dg, H);
  const FxScale sc = fx_scale(kd);
  if (fast) {
    for (int e = threadIdx.x; e < kFfLogN; e += blockDim.x) tab[e] = sc.tab(g_log_tab[e]);
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
        const ulonglong2 mv = fxy[i];
        const FxRest mr = fq[i];
        FxSums a;
        a.clear();
        for (; w.more(); w.step(S)) {
          const ulonglong2 v = fxy[w.k];
          const FxRest r = fq[w.k];
          const fx96 dx = fx_sub(fx96{mv.x, mr.ex}, fx96{v.x, r.ex});
          const fx96 dy = fx_sub(fx96{mv.y, mr.ey}, fx96{v.y, r.ey});
          const uint32_t reach = fx_reach(dx, dy);
          if (reach < fx_cut(r.drop())) {  // or the target itself
            if (w.k != i) {
              PairAcc<double> d;
              pair_free(d, xs[i] - xs[w.k], ys[i] - ys[w.k], qs[w.k]);
              lf += d.lf;
              gx += d.gfx;
              gy += d.gfy;
            }
            continue;
          }
          fx_pair(a, dx, dy, reach, r.q, r.drop(), sc, tab);
        }
        lf += a.log_sum(qe >> 1, sc);
        gx += a.gx(qe >> 1, kd);
        gy += a.gy(qe >> 1, kd);
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
// target: 8.1 ms a call; so 0.74, and 0.17 with the folded M2L and the rest).
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
  static int64_t tab[kFfLogN];
  fx_log_table(tab);
  HP_CUDA(cudaMemcpyToSymbol(g_log_tab, tab, sizeof tab));
  HP_CUDA(prefer_shared(k_prep64));
  HP_CUDA(prefer_shared(k_near64<true>));
  HP_CUDA(prefer_shared(k_near64<false>));
  HP_CUDA(prefer_shared(k_mirror64));
  done[dev] = true;
  return special_init_here();
}

namespace {
// Up to order 28 the integer pairs.  Higher orders, whose truncation lies below the
// rounding of an FP64 sum, and trees of one level, which have no free far field, keep
// the FP64 pairs (1e6 points at order 32: 21.9 ms a step, 6.9 at order 24), which the
// integer ones are compared with point by point.
bool near64_fast(const hpfmm_plan *pl) { return pl->p <= 28 && pl->H >= 2; }
}  // namespace

// Blocks per SM of the integer kernel, which loops over the targets: the far
// field's kernels, bound by the FP64 pipe with few warps, find room beside them
// (the step above with 5, 6, 7, 8 blocks: 3.14, 3.12, 3.16, 3.27 ms).
constexpr int kNearBlocks = 6;

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
                                                          pl->qexp, (ulonglong2 *)pl->fxy,
                                                          (FxRest *)pl->fq);
    const unsigned most = (unsigned)(kNearBlocks * pl->sms);
    k_near64<true><<<nb < most ? nb : most, 128, 0, st>>>(pl->xs, pl->ys, qs, (const ulonglong2 *)pl->fxy,
                                       (const FxRest *)pl->fq, pl->keys, pl->leaf_start, n, pl->H,
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
