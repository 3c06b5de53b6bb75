// row_generic_f32.cu -- the two-stage row forward pass with runtime radices for F32 residuals.
#include "row_generic.cuh"
#include "internal.h"

namespace prnu {

void (*row_forward2_f32(bool big))(PassArgs, const float*, int, float2*) {
  return big ? k_row_forward2<kF32, true, 3> : k_row_forward2<kF32, false, 5>;
}

}  // namespace prnu
