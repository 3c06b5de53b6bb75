// search.cu -- kernels of the EIS-inversion grid search (Sec. 3.2) and their launchers.
//
// Per candidate (frame f, fingerprint p, grid node (lambda, theta)) the fused
// path runs four kernels over a wave of candidates:
//   k_row_forward{2,3} (row_generic.cuh): inverse warp of the residual (Eq. 4, bilinear, zero
//                   outside) fused with the row FFT; two real rows share one
//                   complex FFT; output is the packed half spectrum
//                   [H][W/2] complex whose column 0 holds (DC, Nyquist) pairs;
//   k_col         : column FFT, product conj(X^) K0^ with the cached
//                   fingerprint spectrum, inverse column FFT, in place;
//   k_row_inverse{2,3}: inverse row FFT (two rows per complex FFT) and per-row
//                   max / first arg-max / sum of squares of C;
//   k_finalize    : peak over rows, energy outside the cyclic 11x11 window
//                   (the window's rows are recomputed from the spectrum) and
//                   PCE (Eq. 3).
// k_argmax then keeps the best candidate of each (frame, fingerprint).
#include <float.h>
#include <limits.h>
#include <math.h>

#include <algorithm>

#include "internal.h"
#include "search_common.cuh"

namespace prnu {

// ---------------------------------------------------------------- kernels

// Column pass over a strip of 1 << col_log2 columns of one candidate's packed
// spectrum.  grid = (ceil((W/2) >> lg), wave), block = T.
// mode 0: fwd FFT, x conj(.) * K0^, inv FFT;  1: fwd FFT to out (fingerprint);
// 2: product only;  3: fwd FFT only;  4: inv FFT only (modes 2-4 in place).
__global__ void __launch_bounds__(512, 2) k_col(PassArgs a, int mode, float2* __restrict__ out_f32,
                                              __half2* __restrict__ out_f16, const float* __restrict__ out_scale,
                                              int out_strips) {
  extern __shared__ float2 smem[];
  const int T = blockDim.x, tid = threadIdx.x;
  const int H = a.H, Wh = a.W >> 1;
  const int lg = a.col_log2, NC = 1 << lg;
  const int c0 = blockIdx.x << lg;
  const int slot = blockIdx.y;
  float2* Z = a.spec + (size_t)slot * H * Wh;
  const int n = H << lg;
  float2* buf = smem;
  float2* buf2 = smem + n;
  for (int e = tid; e < n; e += T) {
    const int i = e >> lg, col = c0 + (e & (NC - 1));
    buf[e] = col < Wh ? Z[(size_t)i * Wh + col] : make_float2(0.f, 0.f);
  }
  __syncthreads();
  if (mode == 0 || mode == 1 || mode == 3) {
    float2* r = fft_col<false>(buf, buf2, a.pcol, tid, T, lg);
    if (r != buf) { buf2 = buf; buf = r; }
  }
  if (mode == 1) {
    const float s = out_scale ? *out_scale : 1.f;
    for (int e = tid; e < n; e += T) {
      const int i = e >> lg, col = c0 + (e & (NC - 1));
      if (col >= Wh) continue;
      const float2 v = make_float2(buf[e].x * s, buf[e].y * s);
      const size_t o = fp_index(FpDesc{nullptr, kF32, nullptr, out_strips}, i, col, H, Wh);
      if (out_f16) out_f16[o] = __float22half2_rn(v);
      else out_f32[o] = v;
    }
    return;
  }
  if (mode == 0 || mode == 2) {
    const WorkItem it = item_of(a, slot);
    const FpDesc fp = a.fps[it.fp];
    for (int e = tid; e < n; e += T) {
      const int i = e >> lg, col = c0 + (e & (NC - 1));
      if (col == 0 || col >= Wh) continue;
      const float2 s = load_fp(fp, i, col, H, Wh);
      buf[e] = c_conj_mul(buf[e], s);
    }
    if (c0 == 0) {
      // packed column 0 = DC column + i * Nyquist column of both spectra:
      // separate, take conj(X^) K0^ of each, recombine.
      for (int i = tid; i <= (H >> 1); i += T) {
        const int im = (H - i) % H;
        const float2 F = buf[i << lg], Fm = buf[im << lg];
        const float2 S = load_fp(fp, i, 0, H, Wh), Sm = load_fp(fp, im, 0, H, Wh);
        const float2 A = make_float2(0.5f * (F.x + Fm.x), 0.5f * (F.y - Fm.y));
        const float2 B = make_float2(0.5f * (F.y + Fm.y), 0.5f * (Fm.x - F.x));
        const float2 Ka = make_float2(0.5f * (S.x + Sm.x), 0.5f * (S.y - Sm.y));
        const float2 Kb = make_float2(0.5f * (S.y + Sm.y), 0.5f * (Sm.x - S.x));
        const float2 p1 = c_conj_mul(A, Ka), p2 = c_conj_mul(B, Kb);
        const float2 q1 = c_mulc(A, Ka), q2 = c_mulc(B, Kb);
        buf[i << lg] = make_float2(p1.x - p2.y, p1.y + p2.x);
        buf[im << lg] = make_float2(q1.x - q2.y, q1.y + q2.x);
      }
    }
    __syncthreads();
  }
  if (mode == 0 || mode == 4) buf = fft_col<true>(buf, buf2, a.pcol, tid, T, lg);
  for (int e = tid; e < n; e += T) {
    const int i = e >> lg, col = c0 + (e & (NC - 1));
    if (col < Wh) Z[(size_t)i * Wh + col] = buf[e];
  }
}

// Finalisation (search_common.cuh): window pairs b0 .. b1-1 and the row shares of
// the same numbers of candidate slot `s`, to parts (after the caller's barrier,
// by thread 0).
constexpr int kFinMaxWarps = 16;
__device__ void finalize_parts(const PassArgs& a, int s, const FinPeak& pk, int b0, int b1, float2* smem, double* parts) {
  __shared__ double red[kFinParts][kFinMaxWarps];
  const int T = blockDim.x, t = threadIdx.x;
  const int H = a.H, W = a.W, Wh = W >> 1;
  const RowStat* st = a.stats + (size_t)s * H;
  const float2* Z = a.spec + (size_t)s * H * Wh;
  float2* const bufA = smem;
  float2* const bufB = smem + row_smem_len(W);
  for (int b = b0; b < b1; ++b) {
    if (b < kFinRowParts) part_warp(row_share(st, H, pk.py, b, t, T), t, red[b]);
    const int p = window_pair(pk.py, b, H);
    build_full_row(bufA, Z + (size_t)(2 * p) * Wh, Z + (size_t)(2 * p + 1) * Wh, W, t, T);
    __syncthreads();
    const float2* buf = fft_row<true>(bufA, bufB, a.prow, t, T);
    PairEnergy e;
    for (int x = t; x < W; x += T)
      if (cdist(x, pk.px, W) > kHalfWindow) e.add(buf[rpad(x)]);
    part_warp(e.total(cdist(2 * p, pk.py, H) <= kHalfWindow, cdist(2 * p + 1, pk.py, H) <= kHalfWindow), t,
              red[kFinRowParts + b]);
    __syncthreads();   // the row buffers are free again
  }
  if (t == 0)
    for (int b = b0; b < b1; ++b) {
      if (b < kFinRowParts) parts[b] = part_total(red[b], T >> 5);
      parts[kFinRowParts + b] = part_total(red[kFinRowParts + b], T >> 5);
    }
}

// One block per candidate of the wave.
__global__ void __launch_bounds__(512) k_finalize(PassArgs a) {
  extern __shared__ float2 smem[];
  const FinPeak pk = block_peak(a.stats + (size_t)blockIdx.x * a.H, a.H, a.W, threadIdx.x, blockDim.x,
                                reinterpret_cast<WarpRed*>(smem + 2 * row_smem_len(a.W)));
  double parts[kFinParts];
  finalize_parts(a, blockIdx.x, pk, 0, kFinPairParts, smem, parts);
  if (threadIdx.x == 0) finish_candidate(a, blockIdx.x, pk, parts);
}

// One block per window pair (blockIdx.y) of a candidate; k_finalize_sum ends it.
__global__ void __launch_bounds__(512) k_finalize_part(PassArgs a) {
  extern __shared__ float2 smem[];
  const int s = blockIdx.x, b = blockIdx.y;
  const FinPeak pk = block_peak(a.stats + (size_t)s * a.H, a.H, a.W, threadIdx.x, blockDim.x,
                                reinterpret_cast<WarpRed*>(smem + 2 * row_smem_len(a.W)));
  finalize_parts(a, s, pk, b, b + 1, smem, fin_scratch(a, s, pk.py));
  if (b == 0 && threadIdx.x == 0) park_peak(a, s, pk);
}

// The results of candidates whose parts several blocks computed, a thread each.
__global__ void k_finalize_sum(PassArgs a) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= a.nitems || past_count(a, s, 0)) return;
  const CandResult* r = result_of(a, s);
  const FinPeak pk{r->peak, r->py, r->px};
  double parts[kFinParts];
  const double* p = fin_scratch(a, s, pk.py);
#pragma unroll
  for (int k = 0; k < kFinParts; ++k) parts[k] = p[k];
  finish_candidate(a, s, pk, parts);
}

// Best candidate of each (frame, fingerprint) group g: its items are
// first + k*share (k < count) with first = gstart[g / share] + g % share and
// count = (gstart[g / share + 1] - gstart[g / share]) / share, in ascending
// candidate order (share = 1: contiguous groups).  One block per group (a warp's
// chain of loads over 1681 candidates took 24 us).
__global__ void __launch_bounds__(256) k_argmax(const CandResult* __restrict__ res, const WorkItem* __restrict__ items,
                                                const int* __restrict__ gstart, int ngroups, int share,
                                                prnu_result* __restrict__ out, int H, int W) {
  __shared__ double s_v[8];
  __shared__ int s_i[8];
  const int g = blockIdx.x, f = g / share, t = threadIdx.x;
  const int b = gstart[f] + (g - f * share), n = (gstart[f + 1] - gstart[f]) / share;
  double bv = -INFINITY;
  int bi = INT_MAX;
  for (int k = t; k < n; k += 256) better_d(bv, bi, res[b + k * share].pce, b + k * share);
  warp_maxarg_d(bv, bi);
  if ((t & 31) == 0) {
    s_v[t >> 5] = bv;
    s_i[t >> 5] = bi;
  }
  __syncthreads();
  if (t == 0) {
    for (int w = 1; w < 8; ++w) better_d(bv, bi, s_v[w], s_i[w]);
    out[g] = group_result(res, items, n, bi, H, W);
  }
}

__global__ void k_scatter_all(const CandResult* __restrict__ res, int n, int cmax, double* __restrict__ all) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k < n) all[(size_t)res[k].group * cmax + res[k].cand] = res[k].pce;
}

// sum and sum of squares of K, double partials per block
__global__ void k_fp_partials(const float* __restrict__ K, size_t n, double* __restrict__ partials) {
  __shared__ double s1[32], s2[32];
  double a = 0, b = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const double v = K[i];
    a += v;
    b += v * v;
  }
  a = warp_sum(a);
  b = warp_sum(b);
  if ((threadIdx.x & 31) == 0) { s1[threadIdx.x >> 5] = a; s2[threadIdx.x >> 5] = b; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { a += s1[k]; b += s2[k]; }
    partials[2 * blockIdx.x] = a;
    partials[2 * blockIdx.x + 1] = b;
  }
}

__global__ void k_fp_finish(const double* __restrict__ partials, int nblk, size_t n, int half,
                            float* mean_out, float* scale_out, float* inv_scale_out) {
  // one warp: a fixed-order sum per lane, then across the lanes (a single
  // thread's chain of 256 dependent loads and FP64 adds took 27 us)
  double a = 0, b = 0;
  for (int k = threadIdx.x; k < nblk; k += 32) { a += partials[2 * k]; b += partials[2 * k + 1]; }
  a = warp_sum(a);
  b = warp_sum(b);
  if (threadIdx.x != 0) return;
  const double mean = a / (double)n;
  double ss = b - (double)n * mean * mean;          // sum of (K - mean)^2
  if (ss < 0) ss = 0;
  double s = 1.0;
  // FP16 storage: scale the spectrum to unit RMS magnitude (Parseval:
  // mean |K0^|^2 = sum K0^2 for the unnormalised DFT).
  if (half && ss > 0) s = 1.0 / sqrt(ss);
  *mean_out = (float)mean;
  *scale_out = (float)s;
  *inv_scale_out = (float)(1.0 / (double)(float)s);
}

// ---------------------------------------------------------------- naive per-candidate path

__global__ void k_naive_warp(PassArgs a, float* __restrict__ X) {
  const WorkItem it = a.items[a.item0];
  const int H = a.H, W = a.W;
  const size_t base = (size_t)it.frame * H * W;
  const float cx = 0.5f * (float)(W - 1), cy = 0.5f * (float)(H - 1);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < (size_t)H * W;
       i += (size_t)gridDim.x * blockDim.x) {
    const int y = (int)(i / W), x = (int)(i - (size_t)y * W);
    const float dx = (float)x - cx, dy = (float)y - cy;
    const float qx = fmaf(it.a11, dx, fmaf(it.a12, dy, cx));
    const float qy = fmaf(it.a21, dx, fmaf(it.a22, dy, cy));
    X[i] = bilinear<kF32>(a.resid, base, H, W, W, qx, qy);
  }
}

__global__ void k_naive_reduce(const float* __restrict__ C, size_t n, float* bmax, int* barg, double* bsum) {
  __shared__ float sm[32];
  __shared__ int si[32];
  __shared__ double ss[32];
  float v = -INFINITY;
  int vi = INT_MAX;
  double s = 0;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float c = C[i];
    better_f(v, vi, c, (int)i);
    s += (double)c * c;
  }
  warp_maxarg(v, vi);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) { sm[threadIdx.x >> 5] = v; si[threadIdx.x >> 5] = vi; ss[threadIdx.x >> 5] = s; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 1; k < (int)(blockDim.x >> 5); ++k) { better_f(v, vi, sm[k], si[k]); s += ss[k]; }
    bmax[blockIdx.x] = v;
    barg[blockIdx.x] = vi;
    bsum[blockIdx.x] = s;
  }
}

__global__ void k_naive_final(const float* __restrict__ C, int H, int W, const WorkItem* __restrict__ itp,
                              const FpDesc* __restrict__ fps, const float* __restrict__ scale,
                              const float* bmax, const int* barg, const double* bsum, int nblk,
                              CandResult* __restrict__ out) {
  if (threadIdx.x != 0) return;
  float v = -INFINITY;
  int vi = INT_MAX;
  double tot = 0;
  for (int k = 0; k < nblk; ++k) { better_f(v, vi, bmax[k], barg[k]); tot += bsum[k]; }
  if (vi == INT_MAX) vi = 0;
  const int py = vi / W, px = vi - py * W;
  double win = 0;
  for (int dy = -kHalfWindow; dy <= kHalfWindow; ++dy)
    for (int dx = -kHalfWindow; dx <= kHalfWindow; ++dx) {
      const double c = C[(size_t)((py + dy + H) % H) * W + (px + dx + W) % W];
      win += c * c;
    }
  double E = (tot - win) / ((double)H * W - kWindowCount);
  if (E < 0) E = 0;
  const double pk = v;
  double pce;
  if (E > 0.0) pce = (pk < 0 ? -1.0 : 1.0) * pk * pk / E;
  else pce = pk == 0.0 ? 0.0 : (pk < 0 ? -INFINITY : INFINITY);
  const WorkItem it = *itp;
  double pv = pk / ((double)H * W) * (double)(*fps[it.fp].inv_scale);
  if (scale) pv /= (double)scale[it.frame];
  CandResult r;
  r.pce = pce;
  r.peak = (float)pv;
  r.py = py;
  r.px = px;
  r.cand = it.cand;
  r.group = it.group;
  r.pad = 0;
  *out = r;
}

// ---------------------------------------------------------------- launchers

#define PRNU_LAUNCH_CHECK()                                                                 \
  do {                                                                                      \
    cudaError_t e_ = cudaGetLastError();                                                    \
    if (e_ != cudaSuccess) throw Error{PRNU_ECUDA, std::string(__func__) + ": " + cudaGetErrorString(e_)}; \
  } while (0)

void launch_col(const PassArgs& a, int mode, float2* out_f32, void* out_f16, const float* scale, cudaStream_t s,
                LaunchCounter& lc, int out_strips) {
  if (mode == 0 && a.pcol.ra) {
    launch_col2(a, s, lc);
    return;
  }
  int T, maxb;
  col_launch_shape(a.pcol, a.col_log2, &T, &maxb);
  const int Wh = a.W / 2;
  const int nc = 1 << a.col_log2;
  dim3 g((Wh + nc - 1) / nc, a.nitems), b(T);
  const size_t sm = 2 * (size_t)a.H * nc * sizeof(float2);
  __half2* o16 = reinterpret_cast<__half2*>(out_f16);
  ProfScope ps(lc, kKindColumn, s);
  k_col<<<g, b, sm, s>>>(a, mode, out_f32, o16, scale, out_strips);
  PRNU_LAUNCH_CHECK();
  lc.n++;
}

void launch_finalize_sum(const PassArgs& a, cudaStream_t s, LaunchCounter& lc) {
  k_finalize_sum<<<(a.nitems + 63) / 64, 64, 0, s>>>(a);
  PRNU_LAUNCH_CHECK();
  lc.n++;
}

void launch_finalize(const PassArgs& a, cudaStream_t s, LaunchCounter& lc) {
  int T, maxb;
  row_launch_shape(a.prow, &T, &maxb);
  const size_t sm = row_smem_bytes(a.W, 1);
  ProfScope ps(lc, kKindFinalize, s);
  // Up to a candidate per SM the block's chain of six row FFTs is the latency: a
  // block per window pair.  Past that the GPU is full and the peak is searched
  // once (480 x 640, 1764 candidates: 100 against 132 us).
  if (a.nitems <= 152) {
    k_finalize_part<<<dim3(a.nitems, kFinPairParts), T, sm, s>>>(a);
    PRNU_LAUNCH_CHECK();
    launch_finalize_sum(a, s, lc);
  } else {
    k_finalize<<<a.nitems, T, sm, s>>>(a);
    PRNU_LAUNCH_CHECK();
  }
  lc.n++;
}

void launch_argmax(const CandResult* res, const WorkItem* items, const int* group_start, int ngroups, int share,
                   prnu_result* out, const float* /*scale*/, int H, int W, cudaStream_t s, LaunchCounter& lc) {
  if (ngroups <= 0) return;
  ProfScope ps(lc, kKindArgmax, s);
  k_argmax<<<ngroups, 256, 0, s>>>(res, items, group_start, ngroups, std::max(share, 1), out, H, W);
  PRNU_LAUNCH_CHECK();
  lc.n++;
}

void launch_scatter_all(const CandResult* res, int nitems, int cmax, double* all, cudaStream_t s, LaunchCounter& lc) {
  if (nitems <= 0) return;
  ProfScope ps(lc, kKindScatter, s);
  k_scatter_all<<<(nitems + 255) / 256, 256, 0, s>>>(res, nitems, cmax, all);
  PRNU_LAUNCH_CHECK();
  lc.n++;
}

void launch_fp_stats(const float* K, int H, int W, double* partials, int nblk, float* mean_out, float* scale_out,
                     float* inv_scale_out, bool half, cudaStream_t s, LaunchCounter& lc) {
  ProfScope ps(lc, kKindFpSpectrum, s);
  k_fp_partials<<<nblk, 256, 0, s>>>(K, (size_t)H * W, partials);
  PRNU_LAUNCH_CHECK();
  k_fp_finish<<<1, 32, 0, s>>>(partials, nblk, (size_t)H * W, half ? 1 : 0, mean_out, scale_out, inv_scale_out);
  PRNU_LAUNCH_CHECK();
  lc.n += 2;
}

void launch_naive_warp(const PassArgs& a, float* X, cudaStream_t s, LaunchCounter& lc) {
  ProfScope ps(lc, kKindNaiveWarp, s);
  k_naive_warp<<<1024, 256, 0, s>>>(a, X);
  PRNU_LAUNCH_CHECK();
  lc.n++;
}

void launch_naive_pce(const float* C, int H, int W, const WorkItem* item, const FpDesc* fps, const float* scale,
                      CandResult* out, float* bmax, int* barg, double* bsum, int nblk, cudaStream_t s,
                      LaunchCounter& lc) {
  ProfScope ps(lc, kKindNaivePce, s);
  k_naive_reduce<<<nblk, 256, 0, s>>>(C, (size_t)H * W, bmax, barg, bsum);
  PRNU_LAUNCH_CHECK();
  k_naive_final<<<1, 32, 0, s>>>(C, H, W, item, fps, scale, bmax, barg, bsum, nblk, out);
  PRNU_LAUNCH_CHECK();
  lc.n += 2;
}

const char* const kKindNames[kKindCount] = {"residual", "fingerprint_spectrum", "row_forward", "column",
                                             "row_inverse", "finalize", "argmax", "scatter", "naive_warp",
                                             "naive_pce", "fused"};

cudaEvent_t LaunchCounter::take() {
  if (!pool.empty()) {
    cudaEvent_t e = pool.back();
    pool.pop_back();
    return e;
  }
  cudaEvent_t e;
  PRNU_CUDA_TRY(cudaEventCreate(&e));
  return e;
}

void LaunchCounter::start(int kind, cudaStream_t s) {
  std::lock_guard<std::mutex> lk(mu);
  Rec r{kind, take(), take()};
  PRNU_CUDA_TRY(cudaEventRecord(r.a, s));
  recs.push_back(r);
}

void LaunchCounter::stop(cudaStream_t s) {
  std::lock_guard<std::mutex> lk(mu);
  if (!recs.empty()) cudaEventRecord(recs.back().b, s);
}

template <class K>
static void allow_smem(K k) {
  allow_max_dynamic_smem(k);
}

void set_kernel_attributes() {
  allow_smem(k_col);
  allow_smem(k_finalize);
  allow_smem(k_finalize_part);
  allow_col2();
  allow_rows();
  cudaGetLastError();
}

}  // namespace prnu
