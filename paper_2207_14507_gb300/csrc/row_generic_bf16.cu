// row_generic_bf16.cu -- the two-stage row forward pass with runtime radices for BF16 residuals.
#include "row_generic.cuh"
#include "internal.h"

namespace prnu {

void (*row_forward2_bf16(bool big))(PassArgs, const float*, int, float2*) {
  return big ? k_row_forward2<kBF16, true, 3> : k_row_forward2<kBF16, false, 5>;
}

}  // namespace prnu
