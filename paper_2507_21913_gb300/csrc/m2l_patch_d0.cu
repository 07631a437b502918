// m2l_patch_d0.cu -- double-precision instances of the patch free-space M2L for
// p = 2 .. kPatchOrders[0] (see m2l_patch.cuh).
#include "m2l_patch.cuh"

bool m2l_patch_launch_d0(HP_PATCH_ARGS(cd)) {
  return patch_launch_any<double, 2>(
      std::make_integer_sequence<int, kPatchOrders[0] - 1>{}, p, H, lmin, lmax, dg, Tpad, logt, M, A, B, status, st,
      nr, rs, leaf_start, skip_empty);
}
