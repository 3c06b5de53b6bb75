// search_fixed_2160.cu -- the planned kernels of 3840x2160 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_2160() {
  // Rows of 3840 = 16 x 15 x 16 points by 256 threads a row pair, the last radix
  // even so that the row forward's mirror bins come by shuffle.  Registers for 4
  // blocks per SM: row inverse 10.2 us a candidate (5 blocks 10.3, 3 blocks 11.3, 6
  // blocks 12.5; 16 x 16 x 15: 11.2), row forward FP16 17.4 (3 blocks 17.9, 6 blocks
  // 20.9; 16 x 16 x 15: 19.8).
  using D = ShapeDef<Spec<3840, 16, 15, 16>, 256, ColPlan<2160, 48, 45>, Spec<2160, 15, 12, 12>>;
  // us per candidate (FP32 / FP16 fingerprints), 2 blocks per SM: mode 4 - / 18.8,
  // with the L2 prefetch 18.0; mode 2 20.7 / 20.5; mode 1 25.2 / 25.0; mode 0 26
  // (8-column strips, 1 block: 24 to 28).  The three-stage plan: 21.9 (FP16).
  return D::make({D::row<2>(), D::row<1, 4, 4>()},
                 {D::col<4, 2, 4, 152>(), D::col<4, 2, 2, 152>(), D::col<4, 2, 1>(), D::col<4, 2, 0>()},
                 {D::col_fwd<4, 2>(), D::col_inv<4, 2>(), D::col_inv<4, 2, 4>()}, D::persist<256, 2, 4>());
}

}  // namespace prnu
