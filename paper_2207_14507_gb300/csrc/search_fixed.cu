// search_fixed.cu -- registry and launchers of the compile-time-planned kernels
// (search_fixed.cuh): the sizes they exist for, the TMA descriptors of their
// spectra, and the launches of a wave.
#include <cudaTypedefs.h>

#include <algorithm>
#include <mutex>

#include "internal.h"
#include "search_common.cuh"
#include "search_fixed.h"

namespace prnu {

namespace {

std::vector<FixedShape> build_registry() {
  std::vector<FixedShape> v{fixed_shape_1080(), fixed_shape_720(), fixed_shape_2160(), fixed_shape_256()};
  cudaGetLastError();
  return v;
}

}  // namespace

const FixedShape* find_fixed(int H, int W) {
  static std::once_flag once;
  static std::vector<FixedShape> reg;
  std::call_once(once, [] { reg = build_registry(); });
  for (auto& s : reg)
    if (s.H == H && s.W == W) return &s;
  return nullptr;
}

bool fixed_supports(const FixedShape& fs, int H, int ppb) {
  const FixedRow& r = fs.row_for(ppb);
  return (H / 2) % r.ppb == 0;
}

namespace {

// cuTensorMapEncodeTiled from the driver, looked up once (nullptr if absent)
PFN_cuTensorMapEncodeTiled_v12000 tensor_map_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q{};
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(p);
    cudaGetLastError();
  });
  return fn;
}

// The workspace spectra [rows][W/2] float2 as a [rows][W] float tensor with
// boxes of br rows x 2*nc floats (nc complex columns).
bool encode_spec_map(CUtensorMap* m, const float2* base, int W, long long rows, int nc, int br) {
  PFN_cuTensorMapEncodeTiled_v12000 enc = tensor_map_encoder();
  if (!enc || br <= 0) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)W, (cuuint64_t)rows};
  const cuuint64_t strides[1] = {(cuuint64_t)W * sizeof(float)};
  const cuuint32_t box[2] = {(cuuint32_t)(2 * nc), (cuuint32_t)br};
  const cuuint32_t es[2] = {1, 1};
  return enc(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float2*>(base), dims, strides, box, es,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

void launch_fixed_wave(const PassArgs& a, const FixedShape& fs, int col_variant, cudaStream_t s, LaunchCounter& lc) {
  // forward units (several candidates of one frame and node): the row pass
  // and the forward column FFT per unit, into slots a.nitems + u; the product
  // and the inverse column FFT per candidate
  const bool units = a.units != nullptr || a.share > 1;
  const int nunits = units ? a.nunits : a.nitems;
  int v = std::max(0, std::min(col_variant, (int)fs.cols.size() - 1));
  // a variant whose fingerprint region holds FP16 bins only (mode 4) steps
  // aside for FP32 fingerprints
  if (fs.cols[v].mode == 4 && a.fp_f32) v = fs.f32_col;
  // forward units take the split pass, its inverse half in the mode that is
  // fastest for the wave's fingerprints (the bits are the same in all)
  const FixedCol& fc = units ? (fs.col_inv_h.fn && !a.fp_f32 ? fs.col_inv_h : fs.col_inv) : fs.cols[v];
  const FixedRow& fr = fs.row_for(a.pairs_per_block);
  const int Wh = a.W / 2;
  void* args[] = {const_cast<PassArgs*>(&a)};
  alignas(64) CUtensorMap map;
  const long long rows = (long long)(a.nitems + (units ? nunits : 0)) * a.H;
  if (fc.tma && !encode_spec_map(&map, a.spec, a.W, rows, fc.nc, fc.br))
    throw Error{PRNU_ECUDA, "cannot describe the workspace spectra for TMA (cuTensorMapEncodeTiled)"};
  void* targs[] = {const_cast<PassArgs*>(&a), &map};
  {
    ProfScope ps(lc, kKindRowForward, s);
    dim3 g((a.H / 2) / fr.ppb, nunits), b(fr.threads * fr.ppb);
    PRNU_CUDA_TRY(cudaLaunchKernel(fr.fwd[a.rdtype], g, b, args, fr.smem, s));
  }
  auto col_grid = [&](const FixedCol& c, int n) { return dim3((Wh + c.nc - 1) / c.nc, n); };
  if (units) {   // the forward half, per unit (same strip shape as the inverse half: one tensor map)
    ProfScope ps(lc, kKindColumn, s);
    const FixedCol& ff = fs.col_fwd;
    PRNU_CUDA_TRY(cudaLaunchKernel(ff.fn, col_grid(ff, nunits), dim3(ff.threads), targs, ff.smem, s));
    lc.n += 1;
  }
  {
    ProfScope ps(lc, kKindColumn, s);
    PRNU_CUDA_TRY(cudaLaunchKernel(fc.fn, col_grid(fc, a.nitems), dim3(fc.threads), fc.tma ? targs : args, fc.smem,
                                   s));
  }
  {
    ProfScope ps(lc, kKindRowInverse, s);
    dim3 g((a.H / 2) / fr.ppb, a.nitems), b(fr.threads_inv * fr.ppb);
    PRNU_CUDA_TRY(cudaLaunchKernel(fr.inv, g, b, args, fr.smem, s));
  }
  {
    ProfScope ps(lc, kKindFinalize, s);
    PRNU_CUDA_TRY(cudaLaunchKernel(fr.fin, dim3(a.nitems, fr.fin_split ? kFinPairParts : 1), dim3(fr.fin_threads), args,
                                   fr.fin_smem, s));
    if (fr.fin_split) launch_finalize_sum(a, s, lc);
  }
  lc.n += 4;
}

void launch_persistent(const PassArgs& a, const PersistArgs& p, const FixedShape& fs, int sm_count, cudaStream_t s,
                       LaunchCounter& lc) {
  const FixedPersist& f = fs.persist;
  void* args[] = {const_cast<PassArgs*>(&a), const_cast<PersistArgs*>(&p)};
  ProfScope ps(lc, kKindFused, s);
  const int grid = sm_count * f.blocks_per_sm[a.rdtype];
  PRNU_CUDA_TRY(cudaLaunchKernel(f.fn[a.rdtype], dim3(grid), dim3(f.threads), args, f.smem, s));
  lc.n += 1;
}

}  // namespace prnu

