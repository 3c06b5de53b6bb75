// row_generic.cu -- launches of the row passes with runtime radices.
#include "internal.h"
#include "row_generic.cuh"

namespace prnu {

// The radices with the fewest threads a block, then the smallest largest radix.  Every
// even 5-smooth length in [16, 4096] has this or a two-stage plan.
bool row3_radices(int n, int r[3]) {
  static const int radices[] = {5, 8, 9, 10, 12, 15, 16, 18, 20, 25};
  int best = INT_MAX;
  for (int p : radices)
    for (int q : radices)
      for (int s : radices) {
        if (p > q || q > s || p * q * s != n) continue;
        const int c[3] = {p, q, s}, cost = row3_threads(c) * 64 + s;
        if (row3_threads(c) > kRow3MaxThreads || cost >= best) continue;
        best = cost;
        for (int k = 0; k < 3; ++k) r[k] = c[k];
      }
  return best < INT_MAX;
}

using RowForward2 = void (*)(PassArgs, const float*, int, float2*);
RowForward2 row_forward2_f32(bool three);
RowForward2 row_forward2_f16(bool three);
RowForward2 row_forward2_bf16(bool three);

namespace {

struct RowShape {
  bool three;
  dim3 grid;
  int threads;
  size_t smem;
};
RowShape row_shape(const PassArgs& a) {
  const FftPlan& p = a.prow;
  PRNU_CHECK_ARG(p.ra != 0 || p.r3[0] != 0, "row plan");
  if (p.r3[0])
    return {true, dim3(a.H / 2, a.nitems), row3_threads(p.r3), (size_t)row3_points(p.r3) * sizeof(float2)};
  return {false, dim3((a.H / 2 + kRow2Pairs - 1) / kRow2Pairs, a.nitems), kRow2Threads * kRow2Pairs,
          row2_smem(p.ra, p.rb)};
}

}  // namespace

void launch_row_forward(const PassArgs& a, bool warp, const float* mean_sub, float2* out, cudaStream_t s,
                        LaunchCounter& lc) {
  const RowShape r = row_shape(a);
  const RowForward2 fn = a.rdtype == kF32 ? row_forward2_f32(r.three) : a.rdtype == kF16 ? row_forward2_f16(r.three)
                                                                                         : row_forward2_bf16(r.three);
  ProfScope ps(lc, kKindRowForward, s);
  fn<<<r.grid, r.threads, r.smem, s>>>(a, mean_sub, warp ? 1 : 0, out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void launch_row_inverse(const PassArgs& a, float* c_out, cudaStream_t s, LaunchCounter& lc) {
  const RowShape r = row_shape(a);
  ProfScope ps(lc, kKindRowInverse, s);
  (r.three ? k_row_inverse3<2> : k_row_inverse2<5>)<<<r.grid, r.threads, r.smem, s>>>(a, c_out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void allow_rows() {
  for (bool three : {false, true}) {
    allow_max_dynamic_smem(row_forward2_f32(three));
    allow_max_dynamic_smem(row_forward2_f16(three));
    allow_max_dynamic_smem(row_forward2_bf16(three));
  }
  allow_max_dynamic_smem(k_row_inverse2<5>);
  allow_max_dynamic_smem(k_row_inverse3<2>);
}

}  // namespace prnu
