// search_fixed_1080.cu -- the planned kernels of 1920x1080 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_1080() {
  using D = ShapeDef<Spec<1920, 16, 12, 10>, 192, Spec<1080, 9, 12, 10>, 160>;
  return D::make({D::row<2>(), D::row<1, 8>()},
                 {D::col<4, 240, 3, 3>(), D::col<4, 240, 3, 2>(), D::col<4, 240, 3, 1>(),
                  D::col<4, 240, 3, 0>(), D::col<8, 480, 1, 1>()},
                 {D::col_fwd<4, 240, 3>(), D::col_inv<4, 240, 3>(), D::col_inv<4, 240, 3, 3>(),
                  D::col_inv<4, 240, 4, 4>()},
                 D::persist<192, 2, 4>());
}

}  // namespace prnu
