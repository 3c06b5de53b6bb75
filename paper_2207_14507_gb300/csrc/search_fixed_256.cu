// search_fixed_256.cu -- the planned kernels of 256x256 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_256() {
  // Rows of 256 = 16 x 16 points by 16 threads a row pair, eight pairs to a block:
  // every thread holds a butterfly in both stages (32 threads a pair left half of
  // them idle).  Registers for 6 blocks per SM: row inverse 0.078 us a candidate
  // (unbounded 0.101, 8 blocks 0.089; 32 threads 0.131), row forward 0.122 (0.130,
  // 0.128; 32 threads 0.203).
  using D = ShapeDef<Spec<256, 16, 16>, 16, ColPlan<256, 16, 16>, Spec<256, 16, 16>>;
  // us per candidate: 4-column strips, mode 3 with 12 blocks per SM 0.104 (the
  // default); 8-column strips, mode 1 with 8 blocks 0.109, mode 2 0.109, mode 3 0.110;
  // 16-column strips, mode 2 0.115, mode 3 0.124.
  return D::make({D::row<8, 6, 6>(), D::row<4>()},
                 {D::col<4, 12, 3>(), D::col<8, 8, 1>(), D::col<16, 4, 2>()},
                 {D::col_fwd<16, 4>(), D::col_inv<16, 3, 3>()},
                 D::persist<32, 8, 16>());
}

}  // namespace prnu
