// row_generic_f32.cu -- the row forward passes with runtime radices for F32 residuals.
#include "row_generic.cuh"
#include "internal.h"

namespace prnu {

void (*row_forward2_f32(bool three))(PassArgs, const float*, int, float2*) {
  return three ? k_row_forward3<kF32> : k_row_forward2<kF32, 5>;
}

}  // namespace prnu
