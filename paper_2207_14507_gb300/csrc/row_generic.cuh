// row_generic.cuh -- the row passes for widths W = RA * RB whose two radices a
// thread can hold, chosen at run time (the other widths take the ping-pong
// stages of search.cu).
//
// A row pair (two real rows as one complex transform) belongs to a group of
// one warp (radices up to 32) or two (up to 48):
//   stage A : thread t < RB reads x[t + r RB], r < RA; writes t LA + r (LA odd:
//             distinct banks for the lanes)
//   stage B : thread t < RA reads x[t + r RA], twiddle w_W^(rt); leaves outputs
//             t + r RA in its registers
// so the row crosses shared memory once between the stages, every address is a
// base plus a multiple of one stride, and a group of one warp needs no block
// barrier.  The three ping-pong stages spent 153 warp instructions a complex
// point on their indices (58 in the compile-time plans).  Microseconds a
// candidate (row forward, row inverse): 480 x 640 1.37, 1.20 -> 0.84, 0.53; 540 x
// 960 2.84, 2.40 -> 1.35, 0.72; 900 x 1600 6.67, 5.25 -> 6.13, 3.77.
#pragma once
#include "col_generic.cuh"

namespace prnu {

// threads of a row pair and row pairs of a block (a block of 128 threads)
__host__ __device__ constexpr int row2_threads(bool big) { return big ? 64 : 32; }
__host__ __device__ constexpr int row2_pairs(bool big) { return big ? 2 : 4; }
__host__ __device__ constexpr size_t row2_smem(int ra, int rb, bool big) {
  return (size_t)row2_pairs(big) * ((size_t)rb * odd_pitch(ra) * sizeof(float2));
}

template <bool BIG>
__device__ __forceinline__ void group_sync() {
  if (BIG) __syncthreads();
  else __syncwarp();
}

// The warped residual (WARP of blockIdx.y's item) or the image at a.resid
// minus *mean_sub (a.items null), two rows to a group, and its row FFT's
// packed half spectra.  grid = (ceil((H/2) / pairs), candidates).
template <int DT, bool BIG, int MINB>
__global__ void __launch_bounds__(128, MINB) k_row_forward2(PassArgs a, const float* __restrict__ mean_sub, int warp,
                                                            float2* __restrict__ out_override) {
  extern __shared__ float2 smem[];
  constexpr int T = row2_threads(BIG), PPB = row2_pairs(BIG);
  const int grp = threadIdx.x / T, t = threadIdx.x - grp * T;
  const int H = a.H, W = a.W, Wh = W >> 1, ra = a.prow.ra, rb = a.prow.rb;
  const int pair = blockIdx.x * PPB + grp, slot = blockIdx.y;
  const bool active = pair < (H >> 1);
  float2* sm = smem + (size_t)grp * rb * odd_pitch(ra);
  const int y0 = 2 * pair;
  if (active) {
    if (warp) {
      const WorkItem it = item_of(a, slot);
      size_t base;
      const void* Rf = frame_of(a, it.frame, &base);
      const float cx = 0.5f * (float)(W - 1), cy = 0.5f * (float)(H - 1);
      const float dy0 = (float)y0 - cy, dy1 = (float)(y0 + 1) - cy;
      const float bx0 = fmaf(it.a12, dy0, cx), by0 = fmaf(it.a22, dy0, cy);
      const float bx1 = fmaf(it.a12, dy1, cx), by1 = fmaf(it.a22, dy1, cy);
#pragma unroll 2
      for (int x = t; x < W; x += T) {
        const float dx = (float)x - cx;
        sm[x] = make_float2(bilinear<DT>(Rf, base, H, W, a.rpitch, fmaf(it.a11, dx, bx0), fmaf(it.a21, dx, by0)),
                            bilinear<DT>(Rf, base, H, W, a.rpitch, fmaf(it.a11, dx, bx1), fmaf(it.a21, dx, by1)));
      }
    } else {
      const float m = mean_sub ? *mean_sub : 0.f;
      for (int x = t; x < W; x += T)
        sm[x] = make_float2(load_store_type<DT>(a.resid, (size_t)y0 * W + x) - m,
                            load_store_type<DT>(a.resid, (size_t)(y0 + 1) * W + x) - m);
    }
  }
  group_sync<BIG>();
  with_radix<BIG>(ra, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    float2 u[R];
    if (t < rb) {
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = sm[t + r * rb];
    }
    group_sync<BIG>();
    if (t < rb) {
      DftP<R, false>::run(u);
      float2* dst = sm + t * odd_pitch(R);
#pragma unroll
      for (int r = 0; r < R; ++r) dst[r] = u[r];
    }
  });
  group_sync<BIG>();
  with_radix<BIG>(rb, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    float2 v[R];
    if (t < ra) {
      const int step = odd_pitch(ra);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = sm[t + r * step];
      plan_twiddles<R, false>(v, t, ra, a.tw + a.prow.tw_fwd);
      DftP<R, false>::run(v);
    }
    group_sync<BIG>();
    if (t < ra) {
#pragma unroll
      for (int r = 0; r < R; ++r) sm[t + r * ra] = v[r];
    }
  });
  group_sync<BIG>();
  if (active) {
    float2* o0 = (out_override ? out_override : a.spec + (size_t)slot * H * Wh) + (size_t)y0 * Wh;
    float2* o1 = o0 + Wh;
#pragma unroll 4
    for (int k = t; k < Wh; k += T) {
      const float2 zk = sm[k], zm = sm[k == 0 ? Wh : W - k];
      o0[k] = k == 0 ? make_float2(zk.x, zm.x) : make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
      o1[k] = k == 0 ? make_float2(zk.y, zm.y) : make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
    }
  }
}

// The inverse row FFT of two rows per group, and per-row max / first arg-max /
// sum of squares into a.stats, or (c_out) the rows themselves.
template <bool BIG, int MINB>
__global__ void __launch_bounds__(128, MINB) k_row_inverse2(PassArgs a, float* __restrict__ c_out) {
  extern __shared__ float2 smem[];
  __shared__ RowRed s_red[2][2];
  constexpr int T = row2_threads(BIG), PPB = row2_pairs(BIG);
  const int grp = threadIdx.x / T, t = threadIdx.x - grp * T;
  const int H = a.H, W = a.W, Wh = W >> 1, ra = a.prow.ra, rb = a.prow.rb;
  const int pair = blockIdx.x * PPB + grp, slot = blockIdx.y;
  const bool active = pair < (H >> 1);
  float2* sm = smem + (size_t)grp * rb * odd_pitch(ra);
  const float2* pa = a.spec + ((size_t)slot * H + 2 * (active ? pair : 0)) * Wh;
  const float2* pb = pa + Wh;
  with_radix<BIG>(ra, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    if (t >= rb) return;
    float2 u[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      // bin i of z = G_a + i G_b from the packed half spectra (bin 0 holds DC and
      // Nyquist, both real)
      const int i = t + r * rb;
      const bool up = i > Wh;
      const int k = up ? W - i : i == Wh ? 0 : i;
      const float2 A = __ldg(pa + k), B = __ldg(pb + k);
      const float sg = up ? -1.f : 1.f;
      u[r] = make_float2(fmaf(-sg, B.y, A.x), fmaf(sg, A.y, B.x));
      if (i == 0) u[r] = make_float2(A.x, B.x);
      if (i == Wh) u[r] = make_float2(A.y, B.y);
    }
    DftP<R, true>::run(u);
    float2* dst = sm + t * odd_pitch(R);
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r] = u[r];
  });
  group_sync<BIG>();
  float ma = -INFINITY, mb = -INFINITY;
  int ia = INT_MAX, ib = INT_MAX;
  float2 sq = make_float2(0.f, 0.f);
  with_radix<BIG>(rb, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    if (t >= ra) return;
    float2 v[R];
    const int step = odd_pitch(ra);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = sm[t + r * step];
    plan_twiddles<R, true>(v, t, ra, a.tw + a.prow.tw_fwd);
    DftP<R, true>::run(v);
    if (c_out) {
      if (!active) return;
      float* oa = c_out + (size_t)(2 * pair) * W;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        oa[t + r * ra] = v[r].x;
        oa[W + t + r * ra] = v[r].y;
      }
      return;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {   // in increasing x: only a larger value moves the arg-max
      const int x = t + r * ra;
      if (v[r].x > ma) {
        ma = v[r].x;
        ia = x;
      }
      if (v[r].y > mb) {
        mb = v[r].y;
        ib = x;
      }
      sq = __ffma2_rn(v[r], v[r], sq);
    }
  });
  if (c_out) return;
  __syncwarp();
  const int ka = __reduce_max_sync(0xffffffffu, float_key(ma));
  const int kb = __reduce_max_sync(0xffffffffu, float_key(mb));
  ia = __reduce_min_sync(0xffffffffu, float_key(ma) == ka ? ia : INT_MAX);
  ib = __reduce_min_sync(0xffffffffu, float_key(mb) == kb ? ib : INT_MAX);
#pragma unroll
  for (int o = 16; o; o >>= 1) {
    sq.x += __shfl_xor_sync(0xffffffffu, sq.x, o);
    sq.y += __shfl_xor_sync(0xffffffffu, sq.y, o);
  }
  RowStat* st = a.stats + (size_t)slot * H + 2 * pair;
  const RowRed red{key_float(ka), ia, key_float(kb), ib, sq.x, 0.f, sq.y, 0.f};
  if constexpr (BIG) {
    if ((t & 31) == 0) s_red[grp][t >> 5] = red;
    __syncthreads();
    if (t == 0 && active) row_stats_final(s_red[grp], 2, st);
  } else if (t == 0 && active) {
    row_stats_final(&red, 1, st);
  }
}

}  // namespace prnu
