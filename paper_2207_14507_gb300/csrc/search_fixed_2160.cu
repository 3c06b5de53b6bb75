// search_fixed_2160.cu -- the planned kernels of 3840x2160 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_2160() {
  using D = ShapeDef<Spec<3840, 16, 16, 15>, 256, Spec<2160, 15, 12, 12>>;
  return D::make({D::row<2>(), D::row<1, 5>()},
                 {D::col<4, 360, 2, 4>(), D::col<4, 360, 2, 2>(), D::col<4, 360, 2, 1>(),
                  D::col<4, 360, 2, 0>()},
                 {D::col_fwd<4, 360, 2>(), D::col_inv<4, 360, 2>(), D::col_inv<4, 360, 2, 4>()},
                 D::persist<256, 2, 4>());
}

}  // namespace prnu
