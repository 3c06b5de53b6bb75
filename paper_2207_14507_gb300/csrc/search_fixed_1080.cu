// search_fixed_1080.cu -- the planned kernels of 1920x1080 frames.
#include "search_fixed.cuh"

namespace prnu {

FixedShape fixed_shape_1080() {
  // Rows of 1920 = 16 x 15 x 8 points by 128 threads a row pair: 120, 128 and
  // 2 x 120 butterflies, where 16 x 12 x 10 by 192 threads left 72 of them idle
  // in the warp's gathers.  Row forward 4.71 -> 4.18 us a candidate (FP32; FP16
  // 4.30 -> 3.68), row inverse 2.50 -> 2.30.  Registers for 8 blocks per SM each:
  // the row inverse takes 2.46 unbounded (50 registers, 10 blocks), 2.33 for 7,
  // the row forward 4.43 unbounded, 4.17 for 7, 4.30 for 9.
  using D = ShapeDef<Spec<1920, 16, 15, 8>, 128, ColPlan<1080, 36, 30>, Spec<1080, 9, 12, 10>>;
  // us per candidate of the column variants (FP32 / FP16 fingerprints): 4-column
  // strips, mode 4 with 4 blocks per SM - / 3.40; mode 1 with 4 blocks 3.72 /
  // 3.58 (3 blocks 4.02 / 4.00); mode 2 with 4 blocks 3.75 / 3.74 (3 blocks 3.89 /
  // 3.93); mode 3 with 3 blocks 3.82 / 3.89; mode 0 4.79; 8-column strips 7.2 (mode
  // 1, 1 block), 3.72 (mode 4, 2 blocks, FP16).  Three stages with the fingerprint
  // by 32-byte TMA rows: 5.38 / 5.30.
  // The persistent launch: three row pairs to a block, 29.3 us a candidate (FP32; FP16
  // 28.8); 16 x 12 x 10 by 192 threads, two pairs, spills 2.4 KB a thread and takes 39.6.
  FixedShape s = D::make({D::row<2>(), D::row<1, 8, 8>()},
                         {D::col<4, 4, 4>(), D::col<4, 4, 2>(), D::col<4, 4, 1>(), D::col<4, 3, 0>(), D::col<8, 1, 1>(),
                          D::col<4, 3, 3>()},
                         {D::col_fwd<4, 4>(), D::col_inv<4, 3, 3>(), D::col_inv<4, 4, 4>()},
                         D::persist<128, 3, 4>());
  s.f32_col = 2;
  return s;
}

}  // namespace prnu
