// search_fixed_720.cu -- the planned kernels of 1280x720 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_720() {
  using D = ShapeDef<Spec<1280, 16, 10, 8>, 160, Spec<720, 9, 10, 8>>;
  return D::make({D::row<2>(), D::row<1>()},
                 {D::col<8, 360, 2, 3>(), D::col<8, 360, 2, 1>(), D::col<8, 360, 2, 2>(),
                  D::col<8, 360, 2, 0>(), D::col<4, 180, 4, 2>(), D::col<8, 360, 3, 4>()},
                 {D::col_fwd<4, 180, 4>(), D::col_inv<4, 180, 4>(), D::col_inv<4, 180, 4, 3>(),
                  D::col_inv<4, 180, 5, 4>()},
                 D::persist<160, 2, 4>());
}

}  // namespace prnu
