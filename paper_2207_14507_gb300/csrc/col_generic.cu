// col_generic.cu -- launches of the two-stage column pass with runtime radices.
#include "col_generic.cuh"
#include "internal.h"

namespace prnu {

namespace {

// Columns per block: 8 up to radix 32 (64 to 256 threads), 4 above (144 to 192).
constexpr int kNC = 8, kNCBig = 4;
using Kernel = void (*)(PassArgs);
const Kernel kSmall = k_col2<kNC, false, 256, 2>;
const Kernel kBig = k_col2<kNCBig, true, 192, 2>;

}  // namespace

// One block size and two register budgets serve all radices: up to 32 at 128
// registers, up to 48 at 168.
bool col2_radices(int n, int* ra, int* rb) {
  static const int radices[] = {3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48};
  int best = 0;
  for (int r : radices) {
    if (n % r) continue;
    for (int q : radices)
      if (r >= q && r * q == n && (best == 0 || r < best)) best = r;
  }
  if (best == 0 || (best > 32 && n / best < 25)) return false;
  *ra = best;
  *rb = n / best;
  return true;
}

void launch_col2(const PassArgs& a, cudaStream_t s, LaunchCounter& lc) {
  const bool big = a.pcol.ra > 32;
  const int nc = big ? kNCBig : kNC;
  const dim3 g((a.W / 2 + nc - 1) / nc, a.nitems), b(col2_threads(a.pcol.ra, a.pcol.rb, nc));
  const size_t sm = (size_t)col2_rows(a.pcol.ra, a.pcol.rb) * nc * sizeof(float2);
  ProfScope ps(lc, kKindColumn, s);
  (big ? kBig : kSmall)<<<g, b, sm, s>>>(a);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void allow_col2() {
  allow_max_dynamic_smem(kSmall);
  allow_max_dynamic_smem(kBig);
}

}  // namespace prnu
