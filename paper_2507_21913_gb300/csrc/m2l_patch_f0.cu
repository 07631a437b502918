// m2l_patch_f0.cu -- single-precision instances of the patch free-space M2L for
// p = 2 .. kPatchOrders[0] (see m2l_patch.cuh).
#include "m2l_patch.cuh"

bool m2l_patch_launch_f0(HP_PATCH_ARGS(cf)) {
  return patch_launch_any<float, 2>(
      std::make_integer_sequence<int, kPatchOrders[0] - 1>{}, p, H, lmin, lmax, dg, Tpad, logt, M, A, B, status, st,
      nr, rs, leaf_start, skip_empty);
}
