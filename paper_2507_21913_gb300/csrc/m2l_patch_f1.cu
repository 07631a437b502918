// m2l_patch_f1.cu -- single-precision instances of the patch free-space M2L for
// p = kPatchOrders[0] + 1 .. kPatchOrders[1] (see m2l_patch.cuh).
#include "m2l_patch.cuh"

bool m2l_patch_launch_f1(HP_PATCH_ARGS(cf)) {
  return patch_launch_any<float, kPatchOrders[0] + 1>(
      std::make_integer_sequence<int, kPatchOrders[1] - kPatchOrders[0]>{}, p, H, lmin, lmax, dg, Tpad, logt, M, A, B, status, st,
      nr, rs, leaf_start, skip_empty);
}
