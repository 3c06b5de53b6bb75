// search_fixed_256.cu -- the planned kernels of 256x256 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_256() {
  using D = ShapeDef<Spec<256, 16, 16>, 32, ColPlan<256, 16, 16>, Spec<256, 16, 16>>;
  // us per candidate (FP32): 8-column strips, mode 1 with 8 blocks per SM 0.115 (the
  // default); 16-column strips, mode 2 0.121, mode 3 0.123, mode 0 0.122.
  FixedShape s = D::make({D::row<4>(), D::row<2>()},
                         {D::col<16, 4, 2>(), D::col<8, 8, 1>(), D::col<16, 3, 3>()},
                         {D::col_fwd<16, 4>(), D::col_inv<16, 4>(), D::col_inv<16, 3, 3>()},
                         D::persist<32, 8, 16>());
  s.default_col = 1;
  return s;
}

}  // namespace prnu
