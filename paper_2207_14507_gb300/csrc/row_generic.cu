// row_generic.cu -- launches of the two-stage row passes with runtime radices.
#include "internal.h"
#include "row_generic.cuh"

namespace prnu {

using RowForward2 = void (*)(PassArgs, const float*, int, float2*);
RowForward2 row_forward2_f32(bool big);
RowForward2 row_forward2_f16(bool big);
RowForward2 row_forward2_bf16(bool big);

namespace {

bool row2_big(const PassArgs& a) { return a.prow.ra > 32; }
dim3 row2_grid(const PassArgs& a) {
  const int n = row2_pairs(row2_big(a));
  return dim3((a.H / 2 + n - 1) / n, a.nitems);
}

}  // namespace

void launch_row_forward2(const PassArgs& a, bool warp, const float* mean_sub, float2* out, cudaStream_t s,
                         LaunchCounter& lc) {
  const bool big = row2_big(a);
  const RowForward2 fn = a.rdtype == kF32 ? row_forward2_f32(big) : a.rdtype == kF16 ? row_forward2_f16(big)
                                                                                     : row_forward2_bf16(big);
  ProfScope ps(lc, kKindRowForward, s);
  fn<<<row2_grid(a), 128, row2_smem(a.prow.ra, a.prow.rb, big), s>>>(a, mean_sub, warp ? 1 : 0, out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void launch_row_inverse2(const PassArgs& a, float* c_out, cudaStream_t s, LaunchCounter& lc) {
  const bool big = row2_big(a);
  ProfScope ps(lc, kKindRowInverse, s);
  (big ? k_row_inverse2<true, 3> : k_row_inverse2<false, 5>)<<<row2_grid(a), 128, row2_smem(a.prow.ra, a.prow.rb, big), s>>>(
      a, c_out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void allow_row2() {
  for (bool big : {false, true}) {
    allow_max_dynamic_smem(row_forward2_f32(big));
    allow_max_dynamic_smem(row_forward2_f16(big));
    allow_max_dynamic_smem(row_forward2_bf16(big));
  }
  allow_max_dynamic_smem(k_row_inverse2<false, 5>);
  allow_max_dynamic_smem(k_row_inverse2<true, 3>);
}

}  // namespace prnu
