// row_generic_f16.cu -- the row forward passes with runtime radices for F16 residuals.
#include "row_generic.cuh"
#include "internal.h"

namespace prnu {

void (*row_forward2_f16(bool three))(PassArgs, const float*, int, float2*) {
  return three ? k_row_forward3<kF16> : k_row_forward2<kF16, 5>;
}

}  // namespace prnu
