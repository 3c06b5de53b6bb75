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
  // us per candidate (FP32 / FP16 fingerprints), 2 blocks per SM: mode 2 with the L2
  // prefetch 17.0 / 16.7 (without 19.4 / 18.1), mode 4 with it - / 17.0 (without
  // 18.4); mode 1 20.0 / 18.9; mode 0 22 / 21.  Three stages with the fingerprint by
  // 32-byte TMA rows: 21.9 (FP16).
  return D::make({D::row<2>(), D::row<1, 4, 4>()},
                 {D::col<4, 2, 2, 152>(), D::col<4, 2, 4, 152>(), D::col<4, 2, 1>(), D::col<4, 2, 0>()},
                 {D::col_fwd<4, 2>(), D::col_inv<4, 2, 2>(), D::col_inv<4, 2, 4>()}, D::persist<256, 2, 4>());
}

}  // namespace prnu
