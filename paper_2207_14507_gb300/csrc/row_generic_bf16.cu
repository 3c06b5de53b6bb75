// row_generic_bf16.cu -- the row forward passes with runtime radices for BF16 residuals.
#include "row_generic.cuh"
#include "internal.h"

namespace prnu {

void (*row_forward2_bf16(bool three))(PassArgs, const float*, int, float2*) {
  return three ? k_row_forward3<kBF16> : k_row_forward2<kBF16, 5>;
}

}  // namespace prnu
