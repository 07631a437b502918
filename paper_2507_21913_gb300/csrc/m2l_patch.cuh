// m2l_patch.cuh -- the patch form of the free-space M2L (Eq. truncatedM2Lcoef
// for the log kernel, the classic 2-D form the paper's Remark reduces to),
// shared by the translation units that instantiate it for each expansion
// order (m2l_patch_f0.cu .. m2l_patch_d2.cu).
#pragma once

#include <mutex>
#include <utility>

#include "common.cuh"
#include "special.cuh"

// strides between the right-hand sides of a multi-RHS evaluation (blockIdx.y
// = RHS index): q in charges, m in expansion coefficients, out in doubles of
// the potential (the gradient has twice that)
struct RhsStride {
  int64_t q, m, out;
};

// The instances, by type and range of orders (one translation unit each, so
// that they compile in parallel): single precision up to kPatchOrders[0], up to
// kPatchOrders[1] and the rest, double precision in the same way.  Levels
// lmin .. lmax of a tree with leaf level H; false when the order has no instance
// or its shared memory does not fit.
constexpr int kPatchOrders[2] = {16, 27};
#define HP_PATCH_ARGS(C)                                                                       \
  int p, int H, int lmin, int lmax, const DevGeom *dg, const C *Tpad, const cd *logt, const C *M, \
      C *A, C *B, int *status, cudaStream_t st, int nr, RhsStride rs, const int *leaf_start,   \
      int skip_empty
bool m2l_patch_launch_f0(HP_PATCH_ARGS(cf));
bool m2l_patch_launch_f1(HP_PATCH_ARGS(cf));
bool m2l_patch_launch_f2(HP_PATCH_ARGS(cf));
bool m2l_patch_launch_d0(HP_PATCH_ARGS(cd));
bool m2l_patch_launch_d1(HP_PATCH_ARGS(cd));
bool m2l_patch_launch_d2(HP_PATCH_ARGS(cd));

namespace {

// A block owns a patch of 8 x 4 parent boxes of one level (4 x 2 in the narrow
// form, see below); their four children of each type are its targets, one type a
// warp.  The block stages the source boxes' multipoles around the patch and the
// 40 translation vectors once; then each target gets the 27 V-list offsets of its
// child type.
//
// A class translation in Hankel form is L'_r += sum_k g_{r+k} M'_k with g_j =
// (j-1)! t^-j (scaled).  Offsets that differ by a rotation by i or a reflection
// share their vector: g_j(i t) = i^-j g_j(t), g_j(conj t) = conj g_j(t).  So the
// sources of one orbit {i^m t, i^m conj t} are folded before the product: with
// W_q,k = sum_m i^{-mq} M'_k(i^m t), V_q,k the same over conj t and q = (r+k) mod 4,
//   L'_r += sum_k Re g_{r+k} (W + V)_q,k + i Im g_{r+k} (W - V)_q,k.
// W and V for the four residues are a 4-point Fourier transform of the sources
// (additions only).  The V-list of a child falls into 7 orbits -- the ring at
// distance 2, (2,1) with 8 sources, (2,0) and (2,2) with 4, and on the two far
// sides (3,1) and (3,2) with 4, (3,0) with 2, (3,3) -- so 26 (p+1) + 152 real
// operations per moment order take the place of 27 * 4 (p+1): 2.9 times fewer
// at p = 12, 3.4 times at p = 24.  The additions are exact enough: sums of two to
// eight moments of equal scale.
//
// A chunk of kFoldK orders k is folded in registers and applied to all output
// orders along its anti-diagonals (each g_j one broadcast read per chunk).
// Where the accumulators would not fit (double precision beyond p = 25), the
// output orders are taken in chunks.
//
// Measured (1e6 points, level 8, alone): single precision at p = 13 70 -> 45 us and
// 66 M -> 21 M warp instructions (latency: 43 % of the issue slots), double
// precision at p = 12 levels 2..8 2.87 -> 1.07 ms (the FP64 pipe).
//
// Two forms of the same kernel.  Wide: a warp takes 32 targets of one child type,
// a lane each.  Narrow, for launches of few patches (below kWidePatches): a warp
// takes 8 targets, four lanes each, every lane a quarter of the chunks of source
// orders, their sums combined by shuffles: four times the blocks and a quarter
// of each thread's chain, which is what bounds the small levels (single precision,
// levels 2..7 at p = 13: 43 -> 37 us; double precision, level 5 at p = 24: 2.19 ->
// 0.24 ms).  (A warp per
// orbit instead ran seven different pieces of code once each and waited for
// instructions.)
constexpr int kPatchThreads = 128;
// launches of fewer wide patches than this take the narrow form (see above)
constexpr int kWidePatches = 256;
template <bool kNarrow>
struct PatchDims {
  static constexpr int kX = kNarrow ? 4 : 8, kY = kNarrow ? 2 : 4;  // parents per block
  static constexpr int kSrc = 2 * kX + 4, kRows = 2 * kY + 4;       // source boxes per block
};
// 7 x 7 offset class (dy + 3) * 7 + (dx + 3) -> its index among the 40 far
// classes, -1 for the near 3 x 3
__constant__ signed char c_slot[49] = {
    0,  1,  2,  3,  4,  5,  6,  7,  8,  9,  10, 11, 12, 13, 14, 15, -1, -1, -1, 16, 17, 18, 19, -1, -1,
    -1, 20, 21, 22, 23, -1, -1, -1, 24, 25, 26, 27, 28, 29, 30, 31, 32, 33, 34, 35, 36, 37, 38, 39};

// output orders per pass over the sources (accumulators in registers)
template <typename R>
constexpr int fold_rows(int P1) {
  const int cap = sizeof(R) == 4 ? 41 : 26;
  const int n = (P1 + cap - 1) / cap;
  return (P1 + n - 1) / n;
}

__device__ __forceinline__ int2 rot90(int2 o, int m) {  // o i^m
  for (int e = 0; e < (m & 3); ++e) o = make_int2(-o.y, o.x);
  return o;
}

// residue q of the rotation sums of NA sources a (rotations 0 .. NA - 1), tau =
// -1 where the chunk's first order is 2 mod 4
template <typename R, int NA>
__device__ __forceinline__ void fold4(const cpx<R> (&a)[4], R tau, cpx<R> (&w)[4]) {
  if constexpr (NA == 1) {
#pragma unroll
    for (int q = 0; q < 4; ++q) w[q] = a[0];
  } else {
    const cpx<R> s = NA == 4 ? a[0] + a[2] : a[0], d = NA == 4 ? a[0] - a[2] : a[0];
    const cpx<R> s1 = NA == 4 ? a[1] + a[3] : a[1], d1 = NA == 4 ? a[1] - a[3] : a[1];
    w[0] = mk<R>(fma(tau, s1.x, s.x), fma(tau, s1.y, s.y));
    w[2] = mk<R>(fma(-tau, s1.x, s.x), fma(-tau, s1.y, s.y));
    w[1] = mk<R>(fma(tau, d1.y, d.x), fma(-tau, d1.x, d.y));
    w[3] = mk<R>(fma(-tau, d1.y, d.x), fma(tau, d1.x, d.y));
  }
}

// entries p[0], p[1] (p at an even index of a 16-byte aligned row): one 16-byte
// read in single precision
__device__ __forceinline__ void load_pair(const cf *p, cf &a, cf &b) {
  const float4 v = *reinterpret_cast<const float4 *>(p);
  a = mk(v.x, v.y);
  b = mk(v.z, v.w);
}
__device__ __forceinline__ void load_pair(const cd *p, cd &a, cd &b) {
  a = p[0];
  b = p[1];
}
// entry kk of a row: in single precision an even kk loads the pair and the odd
// one takes its second half
__device__ __forceinline__ void load_order(const cf *p, int kk, cf &v, cf &next) {
  if (kk & 1) v = next;
  else load_pair(p + kk, v, next);
}
__device__ __forceinline__ void load_order(const cd *p, int kk, cd &v, cd &) { v = p[kk]; }

// orders k0 .. k0 + NK - 1 (k0 even) of one orbit, applied to output orders
// R0 .. R1 - 1: NA sources at rotations of t (pa), as many at rotations of
// conj t with HASB (pb, sigma = -1 where their odd residues change sign), the
// vector G of t (complex, or real).  lg: ln|t d| at k0 = 0, else 0.
template <typename R, int R0, int R1, int NA, bool HASB, bool REAL, int NK>
__device__ __forceinline__ void fold_chunk(cpx<R> (&acc)[R1 - R0], const cpx<R> *const (&pa)[4],
                                           const cpx<R> *const (&pb)[4], const cpx<R> *G, int k0,
                                           R tau, R sigma, R lg) {
  cpx<R> P[NK][4], D[NK][4];
  cpx<R> na[4], nb[4];  // single precision: the next order, loaded in pairs
#pragma unroll
  for (int kk = 0; kk < NK; ++kk) {
    cpx<R> a[4], b[4];
#pragma unroll
    for (int m = 0; m < NA; ++m) {
      load_order(pa[m] + k0, kk, a[m], na[m]);
      if constexpr (HASB) load_order(pb[m] + k0, kk, b[m], nb[m]);
    }
    fold4<R, NA>(a, tau, P[kk]);
    if constexpr (HASB) {
      cpx<R> v[4];
      fold4<R, NA>(b, tau, v);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const R sg = (q & 1) ? sigma : R(1);
        const cpx<R> w = P[kk][q];
        P[kk][q] = mk<R>(fma(sg, v[q].x, w.x), fma(sg, v[q].y, w.y));
        D[kk][q] = mk<R>(fma(-sg, v[q].x, w.x), fma(-sg, v[q].y, w.y));
      }
    }
  }
  // M_0 ln|t d| of every source on Re L_0 (L_0 = -L'_0, M'_0 = M_0)
  if constexpr (R0 == 0) acc[0].x = fma(-lg, P[0][0].x, acc[0].x);
  const cpx<R> *Gk = G + k0;
#pragma unroll
  for (int j = R0 & ~1; j <= R1 + NK - 2; j += 2) {
    cpx<R> g[2];
    load_pair(Gk + j, g[0], g[1]);
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int kk = 0; kk < NK; ++kk) {
        const int r = j + h - kk;
        if (r < R0 || r >= R1) continue;
        const int q = (j + h) & 3;
        if constexpr (HASB) {
          acc[r - R0].x = fma(g[h].x, P[kk][q].x, fma(-g[h].y, D[kk][q].y, acc[r - R0].x));
          acc[r - R0].y = fma(g[h].x, P[kk][q].y, fma(g[h].y, D[kk][q].x, acc[r - R0].y));
        } else if constexpr (REAL) {
          acc[r - R0].x = fma(g[h].x, P[kk][q].x, acc[r - R0].x);
          acc[r - R0].y = fma(g[h].x, P[kk][q].y, acc[r - R0].y);
        } else {
          cfma(acc[r - R0], g[h], P[kk][q]);
        }
      }
  }
}

template <typename R, int P1, int R0, int R1, int NA, bool HASB, bool REAL, bool kNarrow>
__device__ __forceinline__ void fold_orbit(cpx<R> (&acc)[R1 - R0], const cpx<R> *const (&pa)[4],
                                           const cpx<R> *const (&pb)[4], const cpx<R> *G, R sigma,
                                           R lg, int part) {
  // double precision folds 2 orders at a time (registers)
  constexpr int NK = sizeof(R) == 4 ? 4 : 2, TAIL = P1 % NK;
  if constexpr (kNarrow) {
    // chunks part, part + 4, ... of rows padded with zeros to whole chunks
#pragma unroll 1
    for (int k0 = 0; k0 < P1; k0 += 4 * NK) {
      const int k = k0 + part * NK;
      if (k < P1)
        fold_chunk<R, R0, R1, NA, HASB, REAL, NK>(acc, pa, pb, G, k,
                                                  (NK == 2 && (k & 2)) ? R(-1) : R(1), sigma,
                                                  k == 0 ? lg : R(0));
    }
    return;
  }
#pragma unroll 1
  for (int k0 = 0; k0 + NK <= P1; k0 += NK)
    fold_chunk<R, R0, R1, NA, HASB, REAL, NK>(acc, pa, pb, G, k0,
                                              (NK == 2 && (k0 & 2)) ? R(-1) : R(1), sigma,
                                              k0 == 0 ? lg : R(0));
  if constexpr (TAIL > 0)
    fold_chunk<R, R0, R1, NA, HASB, REAL, TAIL>(acc, pa, pb, G, P1 - TAIL,
                                                ((P1 - TAIL) & 2) ? R(-1) : R(1), sigma,
                                                P1 == TAIL ? lg : R(0));
}

// row stride of the staged moments: P1 padded (to whole chunks in the narrow
// form), an odd number of 16-byte units in single precision
template <typename R, int P1, bool kNarrow>
constexpr int patch_stride() {
  const int nk = sizeof(R) == 4 ? 4 : 2;
  const int pp = kNarrow ? (P1 + nk - 1) / nk * nk : (P1 + 1) & ~1;
  return ((pp / 2) & 1) ? pp : pp + 2;
}

// where a target's sources lie in the staged patch
template <typename R, int P1, bool kNarrow>
struct PatchAt {
  const cpx<R> *Mp;
  const unsigned char *sempty;
  int tx, ty;  // the target relative to the patch's first source box
  int part;    // narrow form: the lane's quarter
  static constexpr int PS = patch_stride<R, P1, kNarrow>();
  __device__ __forceinline__ int box(int2 o) const {
    constexpr int W = PatchDims<kNarrow>::kSrc;
    const int col = tx + o.x;
    return (ty + o.y) * W + (col & 1) * (W / 2) + (col >> 1);
  }
  // rotations 0 .. NA - 1 of offset o; false when every source is empty
  template <int NA>
  __device__ __forceinline__ bool sources(int2 o, const cpx<R> *(&p)[4]) const {
    bool any = false;
#pragma unroll
    for (int m = 0; m < NA; ++m) {
      const int b = box(o);
      p[m] = Mp + b * PS;
      any |= !sempty[b];
      o = make_int2(-o.y, o.x);
    }
    return any;
  }
};

__device__ __forceinline__ int class_slot(int2 o) { return c_slot[(o.y + 3) * 7 + (o.x + 3)]; }

// one orbit (0 .. 6, see above) of a target of child type rotation rho
template <typename R, int P1, int R0, int R1, bool kNarrow>
__device__ __forceinline__ void fold_one(int orbit, int rho, const PatchAt<R, P1, kNarrow> &at, const cpx<R> *Ts,
                                         const R *lg, bool skip_empty, cpx<R> (&acc)[R1 - R0]) {
  constexpr int GP = 2 * P1;
  const cpx<R> *pa[4], *pb[4];
  const R sigma = (rho & 1) ? R(-1) : R(1);
  bool any;
  switch (orbit) {
    case 0: {
      const int2 o = make_int2(2, 1);
      any = at.template sources<4>(o, pa);
      any |= at.template sources<4>(make_int2(2, -1), pb);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 4, true, false, kNarrow>(acc, pa, pb, Ts + s * GP, R(1), lg[s], at.part);
      return;
    }
    case 1: {
      const int2 o = make_int2(2, 0);
      any = at.template sources<4>(o, pa);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 4, false, true, kNarrow>(acc, pa, pb, Ts + s * GP, R(1), lg[s], at.part);
      return;
    }
    case 2: {
      const int2 o = make_int2(2, 2);
      any = at.template sources<4>(o, pa);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 4, false, false, kNarrow>(acc, pa, pb, Ts + s * GP, R(1), lg[s], at.part);
      return;
    }
    case 3:
    case 4: {
      const int2 o = rot90(make_int2(3, orbit - 2), rho);
      any = at.template sources<2>(o, pa);
      any |= at.template sources<2>(rot90(make_int2(3, 2 - orbit), rho), pb);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 2, true, false, kNarrow>(acc, pa, pb, Ts + s * GP, sigma, lg[s], at.part);
      return;
    }
    case 5: {
      const int2 o = rot90(make_int2(3, 0), rho);
      any = at.template sources<2>(o, pa);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 2, false, false, kNarrow>(acc, pa, pb, Ts + s * GP, R(1), lg[s], at.part);
      return;
    }
    default: {
      const int2 o = rot90(make_int2(3, 3), rho);
      any = at.template sources<1>(o, pa);
      if (skip_empty && !__any_sync(0xffffffffu, any)) return;
      const int s = class_slot(o);
      fold_orbit<R, P1, R0, R1, 1, false, false, kNarrow>(acc, pa, pb, Ts + s * GP, R(1), lg[s], at.part);
      return;
    }
  }
}

// output orders R0 .. R1 - 1 of a target: its orbits, then the scaled values
// written to A and B
template <typename R, int P1, int R0, bool kNarrow>
__device__ __forceinline__ void fold_rows_of(int rho, const PatchAt<R, P1, kNarrow> &at, bool valid,
                                             bool skip_warp, bool skip_empty, const cpx<R> *Ts,
                                             const R *lg, const R *fac_out, size_t e0,
                                             cpx<R> *__restrict__ A, cpx<R> *__restrict__ B) {
  constexpr int R1 = R0 + fold_rows<R>(P1) < P1 ? R0 + fold_rows<R>(P1) : P1;
  constexpr int NR = R1 - R0;
  const R s = (R)(-0.5 / HP_TWO_PI);
  cpx<R> acc[NR];
#pragma unroll
  for (int r = 0; r < NR; ++r) acc[r] = mk<R>(0, 0);
  if (!skip_warp) {
#pragma unroll 1
    for (int orbit = 0; orbit < 7; ++orbit)
      fold_one<R, P1, R0, R1, kNarrow>(orbit, rho, at, Ts, lg, skip_empty, acc);
  }
  if constexpr (kNarrow) {
#pragma unroll
    for (int r = 0; r < NR; ++r) {
#pragma unroll
      for (int o = 8; o < 32; o <<= 1) {
        acc[r].x += __shfl_xor_sync(0xffffffffu, acc[r].x, o);
        acc[r].y += __shfl_xor_sync(0xffffffffu, acc[r].y, o);
      }
    }
    valid = valid && at.part == 0;
  }
  if (valid) {
#pragma unroll
    for (int r = R0; r < R1; ++r) {
      const cpx<R> v = (s * fac_out[r]) * acc[r - R0];
      A[e0 + r] = v;
      B[e0 + r] = conj(v);
    }
  }
  if constexpr (R1 < P1)
    fold_rows_of<R, P1, R1, kNarrow>(rho, at, valid, skip_warp, skip_empty, Ts, lg, fac_out, e0, A, B);
}

// resident blocks per SM the register allocation aims at: 512 wide blocks (level
// 8) fit in one wave of 4 per SM, not of 3 (orders above 13 would spill)
template <typename R, int P1>
constexpr int patch_min_blocks() {
  return sizeof(R) == 4 ? (P1 <= 14 ? 4 : (P1 <= 21 ? 3 : 2)) : (P1 <= 12 ? 3 : 2);
}

template <typename R, int P1, bool kNarrow>
__global__ void __launch_bounds__(kPatchThreads, patch_min_blocks<R, P1>())
k_m2l_free_patch(int H, int lmin, int lmax, const DevGeom *__restrict__ dg,
                 const cpx<R> *__restrict__ Tpad,
                 const cd *__restrict__ logt, const cpx<R> *__restrict__ M,
                 cpx<R> *__restrict__ A, cpx<R> *__restrict__ B, int *__restrict__ status,
                 RhsStride rs, const int *__restrict__ leaf_start, int skip_empty) {
  M += blockIdx.y * rs.m;
  A += blockIdx.y * rs.m;
  B += blockIdx.y * rs.m;
  // Moments scaled by 16^k/k! when staged, outputs by (-1)^{l+1} 16^l/l!
  // (see the table builder).  Moment rows are padded to an even length PP so
  // that k, k+1 pairs are one 16-byte (single precision) shared-memory load,
  // and so are the (g_j, g_{j+1}) pairs of even j the anti-diagonal walk reads.  The source patch is stored with even columns first, so that the
  // sources of a warp's x-consecutive targets (all of one column parity) are
  // consecutive boxes.  The row stride PS is an odd number of 16-byte units,
  // so that the 8 lanes of a quarter-warp (consecutive source boxes) hit 8
  // different bank groups with their 16-byte (k, k+1) loads.
  constexpr int PS = patch_stride<R, P1, kNarrow>();
  constexpr int GP = 2 * P1;
  using Dims = PatchDims<kNarrow>;
  constexpr int HALF = Dims::kSrc / 2, NSRC = Dims::kSrc * Dims::kRows;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ R fac_in[P1], fac_out[P1];  // 16^k / k!, (-1)^{l+1} 16^l / l!
  __shared__ int sbox[kNarrow ? NSRC : 1];  // source box: its Morton index, -1 outside
  __shared__ unsigned char sempty[NSRC];  // source box holds no point
  cpx<R> *Ts = reinterpret_cast<cpx<R> *>(smem_raw);  // [40][GP], and 4 zeros
  cpx<R> *Mp = Ts + 40 * GP + 4;                       // [kRows][kSrc][PS]
  R *lg = reinterpret_cast<R *>(Mp + NSRC * PS);       // [40] ln|t d|
  // level and patch of this block: kPatch x kPatchRows parents, whose four
  // children of each type are the block's targets (one per thread)
  int b = blockIdx.x, l = lmin;
  for (; l <= lmax; ++l) {
    const int nps = 1 << (l - 1);
    const int npx = nps / Dims::kX < 1 ? 1 : nps / Dims::kX;
    const int npy = nps / Dims::kY < 1 ? 1 : nps / Dims::kY;
    if (b < npx * npy) break;
    b -= npx * npy;
  }
  const int npx = (1 << (l - 1)) / Dims::kX < 1 ? 1 : (1 << (l - 1)) / Dims::kX;
  const int px0 = (b % npx) * Dims::kX, py0 = (b / npx) * Dims::kY;
  const int nparent_side = 1 << (l - 1), nside = 1 << l;
  const int64_t off = level_offset(l);
  const R logd = (R)dg->logd[l];
  // the 40 Hankel vectors by bulk copies (TMA) from the table ([40][2][GP]):
  // copy 0 of each class (16 p + 16 bytes, 16-byte aligned)
  const unsigned tbytes = (unsigned)(sizeof(cpx<R>) * 40 * GP);
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_expect_tx(&bar, tbytes);
    for (int c = 0; c < 40; ++c)
      bulk_g2s(Ts + c * GP, Tpad + (size_t)c * 2 * GP, (unsigned)(sizeof(cpx<R>) * GP), &bar);
  }
  for (int c = threadIdx.x; c < 49; c += blockDim.x)
    if (c_slot[c] >= 0) lg[c_slot[c]] = (R)logt[c].x + logd;
  if (threadIdx.x < P1) {
    double f = 1.0;
    for (int i = 2; i <= (int)threadIdx.x; ++i) f *= (double)i;
    const double r = ldexp(1.0, kHankelLog2R * (int)threadIdx.x);
    fac_in[threadIdx.x] = (R)(r / f);
    fac_out[threadIdx.x] = (R)(((threadIdx.x & 1) ? r : -r) / f);
  }
  if (threadIdx.x < 4) Ts[40 * GP + threadIdx.x] = mk<R>(0, 0);
  __syncthreads();  // fac_in; also publishes the mbarrier initialisation
  // source patch.  Wide: a thread takes a box, P1 independent loads each (fewest
  // instructions: 64 vectors of 500000 at p = 16 took 0.84 ms so, 1.11 ms with the
  // coalesced form).  Narrow: a thread per box finds it, then consecutive threads
  // take consecutive orders (coalesced, the shorter wait).
  const int sx0 = 2 * px0 - 2, sy0 = 2 * py0 - 2;
  const cpx<R> *Ml = M + (size_t)off * P1;
  for (int sb = threadIdx.x; sb < NSRC; sb += kPatchThreads) {
    const int row = sb / Dims::kSrc, colp = sb % Dims::kSrc;  // colp: parity-split column
    const int col = (colp < HALF) ? 2 * colp : 2 * (colp - HALF) + 1;
    const int sx = sx0 + col, sy = sy0 + row;
    int at = -1;
    bool empty = true;
    if (sx >= 0 && sy >= 0 && sx < nside && sy < nside) {
      // points of the box: its leaves are contiguous in Morton order
      const uint64_t mb = box_morton(sx, sy);
      const int sh = 2 * (H - l);
      empty = leaf_start[(mb + 1) << sh] == leaf_start[mb << sh];
      at = (int)mb;
    }
    sempty[sb] = empty ? 1 : 0;
    if constexpr (kNarrow) {
      sbox[sb] = at;
    } else {
      cpx<R> *dst = Mp + (size_t)sb * PS;
      if (at >= 0) {
        cpx<R> v[P1];
#pragma unroll
        for (int k = 0; k < P1; ++k) v[k] = Ml[(size_t)at * P1 + k];
#pragma unroll
        for (int k = 0; k < P1; ++k) dst[k] = fac_in[k] * v[k];
      } else {
#pragma unroll
        for (int k = 0; k < P1; ++k) dst[k] = mk<R>(0, 0);
      }
#pragma unroll
      for (int k = P1; k < PS; ++k) dst[k] = mk<R>(0, 0);
    }
  }
  if constexpr (kNarrow) {
    __syncthreads();
#pragma unroll 4
    for (int e = threadIdx.x; e < NSRC * PS; e += kPatchThreads) {
      const int sb = e / PS, k = e - sb * PS, at = sbox[sb];
      cpx<R> v = mk<R>(0, 0);
      if (at >= 0 && k < P1) v = fac_in[k] * Ml[(size_t)at * P1 + k];
      Mp[e] = v;
    }
  }
  __syncthreads();
  if (!mbar_wait_bounded(&bar, 0)) {
    if (threadIdx.x == 0) atomicOr(status, HPFMM_DEV_TIMEOUT);
    mbar_wait_bounded(&bar, 0);  // give the copy a second bounded chance to land
    return;
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int a = warp & 1, bb = warp >> 1;  // child type handled by this warp
  // the V-list of the type is that of type 0 turned by rho quarter turns
  const int rho = bb ? (a ? 2 : 3) : a;
  const int tl = kNarrow ? lane & 7 : lane;
  const int pxA = px0 + tl % Dims::kX, pyA = py0 + tl / Dims::kX;
  const bool vA = pxA < nparent_side && pyA < nparent_side;
  const int txA = 2 * pxA + a, tyA = 2 * pyA + bb;
  // boxes holding no point need no local expansion (nothing is evaluated in
  // them or below them); a warp whose targets are all empty skips the
  // translations, and so does a warp whose sources of an orbit are all empty
  // (their moments are zero).  Not for evaluation at separate targets, which
  // may lie in empty boxes.
  bool tempty = true;
  if (skip_empty && vA) {
    const int sh = 2 * (H - l);
    const uint64_t mb = box_morton(txA, tyA);
    tempty = leaf_start[(mb + 1) << sh] == leaf_start[mb << sh];
  }
  const bool skip_warp = skip_empty && __all_sync(0xffffffffu, tempty);
  // (lanes beyond a small level's parents read boxes inside the staged patch)
  const PatchAt<R, P1, kNarrow> at{Mp, sempty, txA - sx0, tyA - sy0, lane >> 3};
  const size_t e0 = (size_t)(off + box_morton(vA ? txA : 0, vA ? tyA : 0)) * P1;
  fold_rows_of<R, P1, 0, kNarrow>(rho, at, vA, skip_warp, skip_empty, Ts, lg, fac_out, e0, A, B);
}

template <typename R, int P1, bool kNarrow>
size_t patch_smem() {
  using Dims = PatchDims<kNarrow>;
  return sizeof(cpx<R>) * (40 * 2 * P1 + 4 +
                           Dims::kSrc * Dims::kRows * (size_t)patch_stride<R, P1, kNarrow>()) +
         sizeof(R) * 40;
}

template <bool kNarrow>
int patch_blocks(int lmin, int lmax) {
  using Dims = PatchDims<kNarrow>;
  int nb = 0;
  for (int l = lmin; l <= lmax; ++l) {
    const int nps = 1 << (l - 1);
    nb += (nps / Dims::kX < 1 ? 1 : nps / Dims::kX) * (nps / Dims::kY < 1 ? 1 : nps / Dims::kY);
  }
  return nb;
}

// the kernel's shared-memory limit, set once per device; false when it does
// not fit
template <typename R, int P1, bool kNarrow>
bool patch_ready(size_t &sm) {
  static std::mutex mu;
  static signed char attr[64] = {};  // per device: 0 unknown, 1 set, -1 failed
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return false;
  sm = patch_smem<R, P1, kNarrow>();
  if (sm > 227 * 1024) return false;
  std::lock_guard<std::mutex> lock(mu);
  if (attr[dev] == 0) {
    const bool ok = cudaFuncSetAttribute(k_m2l_free_patch<R, P1, kNarrow>,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)sm) == cudaSuccess &&
                    prefer_shared(k_m2l_free_patch<R, P1, kNarrow>) == cudaSuccess;
    if (!ok) cudaGetLastError();
    attr[dev] = ok ? 1 : -1;
  }
  return attr[dev] > 0;
}

// one order: levels lmin .. lmax in one launch; false when it does not fit
template <typename R, int P1>
bool patch_launch_order(int H, int lmin, int lmax, const DevGeom *dg, const cpx<R> *Tpad,
                        const cd *logt, const cpx<R> *M, cpx<R> *A, cpx<R> *B, int *status,
                        cudaStream_t st, int nr, RhsStride rs, const int *leaf_start,
                        int skip_empty) {
  size_t sm = 0;
  if (lmin < 2) lmin = 2;
  if (lmax < lmin) return patch_ready<R, P1, false>(sm);  // no level to translate
  const int nb = patch_blocks<false>(lmin, lmax);
  if ((int64_t)nb * nr < kWidePatches) {
    if (!patch_ready<R, P1, true>(sm)) return false;
    k_m2l_free_patch<R, P1, true>
        <<<dim3(patch_blocks<true>(lmin, lmax), nr), kPatchThreads, sm, st>>>(
            H, lmin, lmax, dg, Tpad, logt, M, A, B, status, rs, leaf_start, skip_empty);
    return true;
  }
  if (!patch_ready<R, P1, false>(sm)) return false;
  k_m2l_free_patch<R, P1, false><<<dim3(nb, nr), kPatchThreads, sm, st>>>(
      H, lmin, lmax, dg, Tpad, logt, M, A, B, status, rs, leaf_start, skip_empty);
  return true;
}

// the instance of order p among PMIN .. PMIN + sizeof...(Ps) - 1
template <typename R, int PMIN, int... Ps>
bool patch_launch_any(std::integer_sequence<int, Ps...>, int p, int H, int lmin, int lmax,
                      const DevGeom *dg, const cpx<R> *Tpad, const cd *logt, const cpx<R> *M,
                      cpx<R> *A, cpx<R> *B, int *status, cudaStream_t st, int nr, RhsStride rs,
                      const int *leaf_start, int skip_empty) {
  bool r = false;
  (void)((p == PMIN + Ps
              ? (r = patch_launch_order<R, PMIN + Ps + 1>(H, lmin, lmax, dg, Tpad, logt, M, A, B,
                                                          status, st, nr, rs, leaf_start,
                                                          skip_empty),
                 true)
              : false) ||
         ...);
  return r;
}

}  // namespace
