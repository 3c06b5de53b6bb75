// fft_plan.cuh -- block-level FFT stages with a runtime plan (sizes without
// compile-time-planned kernels).
//
// Stages run out of place between two shared-memory buffers (ping-pong): a
// thread loads one butterfly's R inputs, transforms them in registers and
// stores the R outputs before it takes the next butterfly, so no register
// state crosses a barrier.  Two layouts:
//  * row layout: one FFT per block (the finalisation), element i at i + (i >> 4) (one
//    float2 of padding every 16 keeps the strided stores off one bank);
//  * column layout: NC = 1 << lg interleaved FFTs (columns), element i of
//    column c at i*NC + c; butterflies are spread over all threads of the block.
// Twiddles of a stage (R, ns) lie as in TwTab (fft_fixed.cuh): entry (m, k) =
// (w^((2m+1)k), w^((2m+2)k)) with w = exp(-2 pi i / (ns R)) as one float4 at
// m ns + k, so that the threads of a warp, which hold consecutive k, read whole
// cache lines (one table of w_n^k per length, read at stride r, cost up to a
// line per lane and load; 1440 x 2560: row forward 20.9 -> 14.5 us a candidate,
// row inverse 14.5 -> 11.5).
#pragma once
#include "fft_packed.cuh"

namespace prnu {

__device__ __forceinline__ int rpad(int i) { return i + (i >> 4); }
__host__ __device__ constexpr int row_smem_len(int n) { return n + (n >> 4) + 1; }

// v * w (forward) or v * conj(w) (INV), the rounding fixed
template <bool INV>
__device__ __forceinline__ float2 plan_tw_mul(float2 v, float wx, float wy) {
  return INV ? make_float2(__fmaf_rn(v.x, wx, __fmul_rn(v.y, wy)), __fmaf_rn(v.y, wx, -__fmul_rn(v.x, wy)))
             : make_float2(__fmaf_rn(v.x, wx, -__fmul_rn(v.y, wy)), __fmaf_rn(v.x, wy, __fmul_rn(v.y, wx)));
}
template <int R, bool INV>
__device__ __forceinline__ void plan_twiddles(float2 (&v)[R], int k, int ns, const float4* __restrict__ tw) {
#pragma unroll
  for (int m = 0; m < R / 2; ++m) {
    const float4 w = __ldg(tw + m * ns + k);
    v[2 * m + 1] = plan_tw_mul<INV>(v[2 * m + 1], w.x, w.y);
    if (2 * m + 2 < R) v[2 * m + 2] = plan_tw_mul<INV>(v[2 * m + 2], w.z, w.w);
  }
}

// One stage: butterflies j = t, t + T, ..: inputs ld(i), outputs st(i, v).
template <int R, bool INV, class Ld, class St>
__device__ __forceinline__ void plan_stage(const FftPlan& p, int s, int t, int T, Ld&& ld,
                                           St&& st) {
  const int nb = p.n / R, ns = p.ns[s];
  const float4* tw = p.tab + p.tw[s];
  for (int j = t; j < nb; j += T) {
    float2 v[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = ld(j + r * nb);
    int k = 0;
    if (ns > 1) {
      k = j - (int)__umulhi((unsigned)j, p.inv[s]) * ns;
      plan_twiddles<R, INV>(v, k, ns, tw);
    }
    DftP<R, INV>::run(v);
    const int base = (j - k) * R + k;
#pragma unroll
    for (int r = 0; r < R; ++r) st(base + r * ns, v[r]);
  }
}
template <bool INV, class Ld, class St>
__device__ __forceinline__ void plan_stage_any(const FftPlan& p, int s, int t, int T,
                                               Ld&& ld, St&& st) {
  switch (p.radix[s]) {
    case 2: plan_stage<2, INV>(p, s, t, T, ld, st); break;
    case 3: plan_stage<3, INV>(p, s, t, T, ld, st); break;
    case 4: plan_stage<4, INV>(p, s, t, T, ld, st); break;
    case 5: plan_stage<5, INV>(p, s, t, T, ld, st); break;
    case 6: plan_stage<6, INV>(p, s, t, T, ld, st); break;
    case 8: plan_stage<8, INV>(p, s, t, T, ld, st); break;
    case 9: plan_stage<9, INV>(p, s, t, T, ld, st); break;
    case 10: plan_stage<10, INV>(p, s, t, T, ld, st); break;
    case 12: plan_stage<12, INV>(p, s, t, T, ld, st); break;
    case 15: plan_stage<15, INV>(p, s, t, T, ld, st); break;
    default: plan_stage<16, INV>(p, s, t, T, ld, st); break;
  }
}

// The FFT of the data in `a` (row layout), using `b` as the second buffer.  Every
// thread of the block must call it (it holds barriers).  The caller synchronises
// before the call; the result is in the returned buffer and is visible to the
// whole block on return.
template <bool INV>
__device__ float2* fft_row(float2* a, float2* b, const FftPlan& p, int t, int T) {
  for (int s = 0; s < p.nstages; ++s) {
    plan_stage_any<INV>(
        p, s, t, T, [=](int i) { return a[rpad(i)]; }, [=](int i, float2 v) { b[rpad(i)] = v; });
    __syncthreads();
    float2* x = a;
    a = b;
    b = x;
  }
  return a;
}

// The FFTs of the 1 << lg columns in `a` (column layout).
template <bool INV>
__device__ float2* fft_col(float2* a, float2* b, const FftPlan& p, int t, int T, int lg) {
  const int c = t & ((1 << lg) - 1);   // T is a multiple of the columns: a thread keeps its column
  for (int s = 0; s < p.nstages; ++s) {
    plan_stage_any<INV>(
        p, s, t >> lg, T >> lg, [=](int i) { return a[(i << lg) + c]; },
        [=](int i, float2 v) { b[(i << lg) + c] = v; });
    __syncthreads();
    float2* x = a;
    a = b;
    b = x;
  }
  return a;
}

}  // namespace prnu
