// col_generic.cuh -- the column pass for heights H = RA * RB whose two radices a
// thread can hold, chosen at run time: the algorithm of col_pass.cuh (two
// stages each way, one thread per column and butterfly, the strip in groups of
// RA or RB rows at an odd pitch between stages) with the strides and the radix
// as run-time values, the strip loaded and stored by every thread itself.
// Three ping-pong stages each way with runtime radices (k_col) take the other
// heights.  Microseconds a candidate: 480 x 640 2.13 -> 0.62, 900 x
// 1600 10.9 -> 3.5, 1440 x 2560 26.4 -> 12.1, 1500 x 2000 21.5 -> 9.9; latency bounds it
// (12 to 24 warps per SM, strips in 64- or 32-byte rows straight from L2).
#pragma once
#include "common.cuh"
#include "fft_plan.cuh"
#include "search_common.cuh"

namespace prnu {

// The product for the packed column 0 (DC + i*Nyquist columns of two real
// spectra in one complex column): F, Fm the frame bins i and H - i, S, Sm the
// fingerprint bins; unpack both, conj-multiply each real column's spectrum,
// repack.
__device__ __forceinline__ float2 packed_col0_product(float2 F, float2 Fm, float2 S, float2 Sm) {
  const float2 Aa = make_float2(0.5f * (F.x + Fm.x), 0.5f * (F.y - Fm.y));
  const float2 Bb = make_float2(0.5f * (F.y + Fm.y), 0.5f * (Fm.x - F.x));
  const float2 Ka = make_float2(0.5f * (S.x + Sm.x), 0.5f * (S.y - Sm.y));
  const float2 Kb = make_float2(0.5f * (S.y + Sm.y), 0.5f * (Sm.x - S.x));
  const float2 p1 = c_conj_mul(Aa, Ka), p2 = c_conj_mul(Bb, Kb);
  return make_float2(p1.x - p2.y, p1.y + p2.x);
}

__host__ __device__ constexpr int odd_pitch(int r) { return r | 1; }
// rows of the strip buffer
__host__ __device__ constexpr int col2_rows(int ra, int rb) {
  return rb * odd_pitch(ra) > ra * odd_pitch(rb) ? rb * odd_pitch(ra) : ra * odd_pitch(rb);
}
__host__ __device__ constexpr int col2_threads(int ra, int rb, int nc) { return nc * (ra > rb ? ra : rb); }

// The radices of a kernel's switch: each set costs its largest radix' registers.
enum ColSet { kColTo27, kColTo32, kColTo40, kColTo54 };
__host__ __device__ constexpr bool col_set_has(ColSet set, int r) {
  constexpr int lo[] = {3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24}, hi[] = {25, 27, 30, 32, 36, 40, 45, 48, 50, 54};
  const int top = set == kColTo27 ? 27 : set == kColTo32 ? 32 : set == kColTo40 ? 40 : 54;
  if (r > top) return false;
  if (set == kColTo27 || set == kColTo32)
    for (int q : lo)
      if (q == r) return true;
  for (int q : hi)
    if (q == r) return true;
  return false;
}
template <int R>
struct RadixC {
  static constexpr int value = R;
};
// f(R as a compile-time constant); R is in the set (checked before the launch)
template <ColSet SET, class F>
__device__ __forceinline__ void with_radix(int R, F&& f) {
  switch (R) {
#define PRNU_RADIX(r)                                    \
  case r:                                                \
    if constexpr (col_set_has(SET, r)) f(RadixC<r>{});   \
    break;
    PRNU_RADIX(3)
    PRNU_RADIX(4)
    PRNU_RADIX(5)
    PRNU_RADIX(6)
    PRNU_RADIX(8)
    PRNU_RADIX(9)
    PRNU_RADIX(10)
    PRNU_RADIX(12)
    PRNU_RADIX(15)
    PRNU_RADIX(16)
    PRNU_RADIX(18)
    PRNU_RADIX(20)
    PRNU_RADIX(24)
    PRNU_RADIX(25)
    PRNU_RADIX(27)
    PRNU_RADIX(30)
    PRNU_RADIX(32)
    PRNU_RADIX(36)
    PRNU_RADIX(40)
    PRNU_RADIX(45)
    PRNU_RADIX(48)
    PRNU_RADIX(50)
    PRNU_RADIX(54)
#undef PRNU_RADIX
    default: break;
  }
}

template <int NC>
struct Col2 {
  const PassArgs& a;
  float2* sm;
  float2* Z;         // the candidate's spectrum
  const FpDesc& fp;
  int c, j, col;     // column of the strip, butterfly, column of the spectrum

  // forward stage A: rows j + r RB of the spectrum to the strip
  template <int R>
  __device__ __forceinline__ void forward() const {
    const int rb = a.pcol.rb, Wh = a.W >> 1;
    if (j >= rb) return;
    float2 u[R];
    const float2* src = Z + (size_t)j * Wh + col;
    const size_t step = (size_t)rb * Wh;
    const bool in = col < Wh;
#pragma unroll
    for (int r = 0; r < R; ++r) u[r] = in ? __ldg(src + r * step) : make_float2(0.f, 0.f);
    DftP<R, false>::run(u);
    float2* dst = sm + j * odd_pitch(R) * NC + c;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r * NC] = u[r];
  }

  // forward stage B, the product, inverse stage B
  template <int R>
  __device__ __forceinline__ void middle() const {
    const int ra = a.pcol.ra, H = a.H, Wh = a.W >> 1;
    const bool act = j < ra;
    float2 v[R];
    if (act) {
      const float2* src = sm + j * NC + c;
      const int step = odd_pitch(ra) * NC;
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = src[r * step];
      plan_twiddles<R, false>(v, j, ra, a.pcol.tab + a.pcol.tw_fwd);
      DftP<R, false>::run(v);
    }
    __syncthreads();   // every strip value read
    if (col - c == 0) {
      // packed column 0: the product needs bin H - i as well, through two
      // scratch columns in the free strip buffer
      if (c == 0 && act) {
#pragma unroll
        for (int r = 0; r < R; ++r) sm[j + r * ra] = v[r];
      }
      __syncthreads();
      if (c == 0 && act) {
#pragma unroll 1
        for (int i = j; i < H; i += ra) {
          const int im = i == 0 ? 0 : H - i;
          sm[H + i] = packed_col0_product(sm[i], sm[im], load_fp(fp, i, 0, H, Wh), load_fp(fp, im, 0, H, Wh));
        }
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = sm[H + j + r * ra];
      }
      __syncthreads();
    }
    if (!act) return;
    if (col != 0 && col < Wh) {
      const size_t first = fp_index(fp, j, col, H, Wh), step = (size_t)ra * (fp.strips ? 4 : Wh);
      if (fp.dtype == kF32) {
        const float2* s = reinterpret_cast<const float2*>(fp.spec) + first;
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = c_conj_mul(v[r], __ldg(s + r * step));
      } else {
        const __half2* s = reinterpret_cast<const __half2*>(fp.spec) + first;
#pragma unroll
        for (int r = 0; r < R; ++r) v[r] = c_conj_mul(v[r], __half22float2(__ldg(s + r * step)));
      }
    }
    DftP<R, true>::run(v);
    float2* dst = sm + j * odd_pitch(R) * NC + c;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r * NC] = v[r];
  }

  // inverse stage A: the strip to rows j + r RB of the spectrum
  template <int R>
  __device__ __forceinline__ void inverse() const {
    const int rb = a.pcol.rb, Wh = a.W >> 1;
    if (j >= rb) return;
    float2 u[R];
    const float2* src = sm + j * NC + c;
    const int step = odd_pitch(rb) * NC;
#pragma unroll
    for (int r = 0; r < R; ++r) u[r] = src[r * step];
    plan_twiddles<R, true>(u, j, rb, a.pcol.tab + a.pcol.tw_inv);
    DftP<R, true>::run(u);
    if (col >= Wh) return;
    float2* dst = Z + (size_t)j * Wh + col;
    const size_t out = (size_t)rb * Wh;
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r * out] = u[r];
  }
};

// grid = (ceil((W/2) / NC), candidates); block = col2_threads(ra, rb, NC).
template <int NC, ColSet SET, int MAXT, int MINB>
__global__ void __launch_bounds__(MAXT, MINB) k_col2(PassArgs a) {
  extern __shared__ float2 smem[];
  const int c = threadIdx.x % NC, slot = blockIdx.y;
  const WorkItem it = item_of(a, slot);
  const FpDesc fp = a.fps[it.fp];
  const Col2<NC> w{a, smem, a.spec + (size_t)slot * a.H * (a.W >> 1), fp, c, (int)threadIdx.x / NC,
                   (int)blockIdx.x * NC + c};
  with_radix<SET>(a.pcol.ra, [&](auto r) { w.template forward<decltype(r)::value>(); });
  __syncthreads();
  with_radix<SET>(a.pcol.rb, [&](auto r) { w.template middle<decltype(r)::value>(); });
  __syncthreads();
  with_radix<SET>(a.pcol.ra, [&](auto r) { w.template inverse<decltype(r)::value>(); });
}

}  // namespace prnu
