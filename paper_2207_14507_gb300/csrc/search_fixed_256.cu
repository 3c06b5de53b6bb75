// search_fixed_256.cu -- the planned kernels of 256x256 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_256() {
  using D = ShapeDef<Spec<256, 16, 16>, 32, Spec<256, 16, 16>>;
  return D::make({D::row<4>(), D::row<2>()},
                 {D::col<16, 128, 4, 2>(), D::col<16, 128, 4, 0>(), D::col<16, 128, 4, 3>()},
                 {D::col_fwd<16, 128, 4>(), D::col_inv<16, 128, 4>(), D::col_inv<16, 128, 4, 3>()},
                 D::persist<32, 8, 16>());
}

}  // namespace prnu
