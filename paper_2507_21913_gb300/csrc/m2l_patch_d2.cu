// m2l_patch_d2.cu -- double-precision instances of the patch free-space M2L for
// p = kPatchOrders[1] + 1 .. HPFMM_MAX_P (see m2l_patch.cuh).
#include "m2l_patch.cuh"

bool m2l_patch_launch_d2(HP_PATCH_ARGS(cd)) {
  return patch_launch_any<double, kPatchOrders[1] + 1>(
      std::make_integer_sequence<int, HPFMM_MAX_P - kPatchOrders[1]>{}, p, H, lmin, lmax, dg, Tpad, logt, M, A, B, status, st,
      nr, rs, leaf_start, skip_empty);
}
