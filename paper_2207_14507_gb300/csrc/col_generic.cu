// col_generic.cu -- launches of the two-stage column pass with runtime radices.
#include "col_generic.cuh"
#include "internal.h"

namespace prnu {

namespace {

// One kernel for each range of the larger radix, with the blocks per SM (the
// register budget) and columns a block that measured best.  us a candidate:
//   to 27: 4 blocks of 216 threads, 72 registers: 480 x 640 0.62, 540 x 960 1.17, 600 x
//          800 1.07 (3 blocks 0.60, 1.20, 1.11; 5 blocks 0.74, 1.50, 1.67; 128
//          registers, as up to 32, 0.83, 1.44, 1.29)
//   to 32: 2 blocks of 256: 960 x 1000 2.39 (3 blocks 2.54)
//   to 40: 3 blocks of 160: 1296 x 1000 3.70, 1600 x 1000 4.50 (4 blocks 4.00, -; 168
//          registers, as 45 and 48 took, 4.39, 4.96)
//   to 54: 2 blocks of 216: 1500 x 2000 9.9, 2000 x 1500 10.5 (1 block 14.5, 14.4; 3
//          blocks 18.7, 23.9; ping-pong stages 19.6, 28.2), 1920 x 1000 6.0 (at 168 registers 5.9)
struct ColKernel {
  void (*fn)(PassArgs);
  ColSet set;
  int nc, max_threads;
};
template <ColSet SET, int NC, int MAXT, int MINB>
ColKernel col_kernel() {
  return {k_col2<NC, SET, MAXT, MINB>, SET, NC, MAXT};
}
const ColKernel kKernels[] = {col_kernel<kColTo27, 8, 216, 4>(), col_kernel<kColTo32, 8, 256, 2>(),
                              col_kernel<kColTo40, 4, 160, 3>(), col_kernel<kColTo54, 4, 216, 2>()};

}  // namespace

// The smallest larger radix.
bool col2_radices(int n, int* ra, int* rb) {
  static const int radices[] = {3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54};
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
  const int ra = a.pcol.ra, rb = a.pcol.rb;
  const ColKernel& k = kKernels[ra <= 27 ? 0 : ra <= 32 ? 1 : ra <= 40 ? 2 : 3];
  const dim3 g((a.W / 2 + k.nc - 1) / k.nc, a.nitems), b(col2_threads(ra, rb, k.nc));
  PRNU_CHECK_ARG(col_set_has(k.set, ra) && col_set_has(k.set, rb) && (int)b.x <= k.max_threads, "column plan");
  const size_t sm = (size_t)col2_rows(ra, rb) * k.nc * sizeof(float2);
  ProfScope ps(lc, kKindColumn, s);
  k.fn<<<g, b, sm, s>>>(a);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void allow_col2() {
  for (const ColKernel& k : kKernels) allow_max_dynamic_smem(k.fn);
}

}  // namespace prnu
