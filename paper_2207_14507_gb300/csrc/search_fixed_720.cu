// search_fixed_720.cu -- the planned kernels of 1280x720 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_720() {
  // Rows of 1280 = 16 x 10 x 8 points by 80 threads a row pair, two pairs to a
  // block: 80, 128 and 2 x 80 butterflies (160 threads a pair left half of them
  // idle in the warp's gathers).  Registers for 5 blocks per SM: row inverse 1.10
  // us a candidate (unbounded 1.12, 4 blocks 1.15, 7 blocks 1.30; 160 threads 1.33).
  using D = ShapeDef<Spec<1280, 16, 10, 8>, 80, ColPlan<720, 30, 24>, Spec<720, 9, 10, 8>>;
  // us per candidate (FP32 / FP16 fingerprints): 4-column strips, mode 4 with 6
  // blocks per SM - / 1.33 (5 blocks 1.36), mode 2 with 5 blocks 1.45 / 1.42 (4
  // blocks 1.66 / 1.59), mode 3 with 4 blocks 1.49; 8-column strips, mode 4 with 3
  // blocks - / 1.46, mode 2 1.53, mode 3 1.77, mode 1 1.89.
  // The persistent launch: three row pairs of 128 threads to a block, 14.8 us a
  // candidate (FP32 and FP16); 160 threads, two pairs, spills more at 96
  // registers and takes 18.3 (17.6 with scalar butterflies); 8-column strips 18.5.
  FixedShape s = D::make({D::row<2, 5, 5>(), D::row<4>()},
                         {D::col<4, 6, 4>(), D::col<8, 2, 1>(), D::col<4, 5, 2>(), D::col<8, 2, 0>(), D::col<8, 3, 2>(),
                          D::col<4, 4, 3>()},
                         {D::col_fwd<4, 6>(), D::col_inv<4, 4, 3>(), D::col_inv<4, 6, 4>()},
                         D::persist<128, 3, 4>());
  s.f32_col = 2;
  return s;
}

}  // namespace prnu
