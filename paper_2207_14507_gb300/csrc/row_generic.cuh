// row_generic.cuh -- the row passes of widths without compile-time plans: one
// row pair (two real rows as one complex transform) in one shared-memory buffer,
// the radices W = RA * RB or R1 * R2 * R3 chosen at run time.
//
// Two stages, where both radices are at most 32: a warp per row pair,
//   stage A : thread t < RB reads x[t + r RB], r < RA; writes t LA + r (LA odd:
//             distinct banks for the lanes)
//   stage B : thread t < RA reads x[t + r RA], twiddle w_W^(rt); leaves outputs
//             t + r RA in its registers
// so the row crosses shared memory once between the stages, every address is a
// base plus a multiple of one stride, and no block barrier is needed.  The
// ping-pong stages that every width took before spent 153 warp instructions a
// complex point on their indices (58 in the compile-time plans).  Microseconds a
// candidate (row forward, row inverse): 480 x 640 1.37, 1.20 -> 0.84, 0.54; 540 x
// 960 2.84, 2.40 -> 1.35, 0.78.
//
// Three stages for every other even width: a block per row pair, a thread per
// butterfly of the stage that has most, in the same manner (Row3, below).  Two stages
// of radices up to 48 at 168 registers and the ping-pong stages, which took these
// widths, left too few warps for the gathers of the warp (us a candidate, row
// forward, row inverse): 900 x 1600 6.13, 3.77 -> 4.47, 2.65; 1440 x 2560 14.0, 11.5 ->
// 11.9, 7.2; 500 x 4000 11.2, 9.9 -> 8.1, 5.3.  Per pixel the two stages stay ahead
// where they apply (540 x 960: 2.6, 1.5 us a megapixel against 3.1, 1.8 at 900 x 1600).
#pragma once
#include "col_generic.cuh"

namespace prnu {

// threads of a row pair and row pairs of a block of the two-stage kernels
constexpr int kRow2Threads = 32, kRow2Pairs = 4;
__host__ __device__ constexpr size_t row2_smem(int ra, int rb) {
  return (size_t)kRow2Pairs * ((size_t)rb * odd_pitch(ra) * sizeof(float2));
}

// Rows y0, y0 + 1 of the warped residual of item `slot`, or of the image at a.resid
// minus *mean_sub, as the complex sequence sm[0, W).
template <int DT>
__device__ __forceinline__ void load_row_pair(const PassArgs& a, int slot, int y0, const float* __restrict__ mean_sub,
                                              int warp, int t, int T, float2* sm) {
  const int H = a.H, W = a.W;
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

// The packed half spectra of the two rows whose transform lies in sm, to o0 and o0 + Wh.
__device__ __forceinline__ void store_half_spectra(const float2* sm, float2* __restrict__ o0, int W, int t, int T) {
  const int Wh = W >> 1;
  float2* o1 = o0 + Wh;
#pragma unroll 4
  for (int k = t; k < Wh; k += T) {
    const float2 zk = sm[k], zm = sm[k == 0 ? Wh : W - k];
    o0[k] = k == 0 ? make_float2(zk.x, zm.x) : make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
    o1[k] = k == 0 ? make_float2(zk.y, zm.y) : make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
  }
}

// Bins t + r nb (r < R) of z = G_a + i G_b from the packed half spectra pa, pb
// (bin 0 holds DC and Nyquist, both real).
template <int R>
__device__ __forceinline__ void load_full_bins(float2 (&u)[R], const float2* __restrict__ pa,
                                               const float2* __restrict__ pb, int W, int t, int nb) {
  const int Wh = W >> 1;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = t + r * nb;
    const bool up = i > Wh;
    const int k = up ? W - i : i == Wh ? 0 : i;
    const float2 A = __ldg(pa + k), B = __ldg(pb + k);
    const float sg = up ? -1.f : 1.f;
    u[r] = make_float2(fmaf(-sg, B.y, A.x), fmaf(sg, A.y, B.x));
    if (i == 0) u[r] = make_float2(A.x, B.x);
    if (i == Wh) u[r] = make_float2(A.y, B.y);
  }
}

// Maxima, first arg-maxima and sums of squares of a thread's values of two rows,
// its positions met in increasing order.  The squares go to kSums plain FP32
// sums (at most 8 terms each of the 32 a thread can have), which are joined,
// and added up over the warp, in compensated FP32.
struct PairStat {
  static constexpr int kSums = 4;
  float ma = -INFINITY, mb = -INFINITY;
  int ia = INT_MAX, ib = INT_MAX;
  float2 sq[kSums] = {};
  __device__ __forceinline__ void add(int x, int k, float2 v) {   // the thread's k-th value
    if (v.x > ma) {
      ma = v.x;
      ia = x;
    }
    if (v.y > mb) {
      mb = v.y;
      ib = x;
    }
    sq[k % kSums] = __ffma2_rn(v, v, sq[k % kSums]);
  }
  // over the warp
  __device__ __forceinline__ RowRed reduce() {
    __syncwarp();
    const int ka = __reduce_max_sync(0xffffffffu, float_key(ma));
    const int kb = __reduce_max_sync(0xffffffffu, float_key(mb));
    ia = __reduce_min_sync(0xffffffffu, float_key(ma) == ka ? ia : INT_MAX);
    ib = __reduce_min_sync(0xffffffffu, float_key(mb) == kb ? ib : INT_MAX);
    float2 s = sq[0], c = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 1; k < kSums; ++k) csum_add2(s, c, sq[k]);
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      c = __fadd2_rn(c, make_float2(__shfl_xor_sync(0xffffffffu, c.x, o), __shfl_xor_sync(0xffffffffu, c.y, o)));
      csum_add2(s, c, make_float2(__shfl_xor_sync(0xffffffffu, s.x, o), __shfl_xor_sync(0xffffffffu, s.y, o)));
    }
    return RowRed{key_float(ka), ia, key_float(kb), ib, s.x, c.x, s.y, c.y};
  }
};

// The warped residual (`warp`: of blockIdx.y's item) or the image at a.resid
// minus *mean_sub (a.items null), two rows to a warp, and its row FFT's
// packed half spectra.  grid = (ceil((H/2) / pairs), candidates).
template <int DT, int MINB>
__global__ void __launch_bounds__(128, MINB) k_row_forward2(PassArgs a, const float* __restrict__ mean_sub, int warp,
                                                            float2* __restrict__ out_override) {
  extern __shared__ float2 smem[];
  const int grp = threadIdx.x / kRow2Threads, t = threadIdx.x - grp * kRow2Threads;
  const int H = a.H, W = a.W, Wh = W >> 1, ra = a.prow.ra, rb = a.prow.rb;
  const int pair = blockIdx.x * kRow2Pairs + grp, slot = blockIdx.y;
  if (pair >= (H >> 1)) return;
  float2* sm = smem + (size_t)grp * rb * odd_pitch(ra);
  load_row_pair<DT>(a, slot, 2 * pair, mean_sub, warp, t, kRow2Threads, sm);
  __syncwarp();
  with_radix<kColTo32>(ra, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    float2 u[R];
    if (t < rb) {
#pragma unroll
      for (int r = 0; r < R; ++r) u[r] = sm[t + r * rb];
    }
    __syncwarp();
    if (t < rb) {
      DftP<R, false>::run(u);
      float2* dst = sm + t * odd_pitch(R);
#pragma unroll
      for (int r = 0; r < R; ++r) dst[r] = u[r];
    }
  });
  __syncwarp();
  with_radix<kColTo32>(rb, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    float2 v[R];
    if (t < ra) {
      const int step = odd_pitch(ra);
#pragma unroll
      for (int r = 0; r < R; ++r) v[r] = sm[t + r * step];
      plan_twiddles<R, false>(v, t, ra, a.prow.tab + a.prow.tw_fwd);
      DftP<R, false>::run(v);
    }
    __syncwarp();
    if (t < ra) {
#pragma unroll
      for (int r = 0; r < R; ++r) sm[t + r * ra] = v[r];
    }
  });
  __syncwarp();
  store_half_spectra(sm, (out_override ? out_override : a.spec + (size_t)slot * H * Wh) + (size_t)(2 * pair) * Wh, W, t,
                     kRow2Threads);
}

// The inverse row FFT of two rows per warp, and per-row max / first arg-max /
// sum of squares into a.stats, or (c_out) the rows themselves.
template <int MINB>
__global__ void __launch_bounds__(128, MINB) k_row_inverse2(PassArgs a, float* __restrict__ c_out) {
  extern __shared__ float2 smem[];
  const int grp = threadIdx.x / kRow2Threads, t = threadIdx.x - grp * kRow2Threads;
  const int H = a.H, W = a.W, Wh = W >> 1, ra = a.prow.ra, rb = a.prow.rb;
  const int pair = blockIdx.x * kRow2Pairs + grp, slot = blockIdx.y;
  if (pair >= (H >> 1)) return;
  float2* sm = smem + (size_t)grp * rb * odd_pitch(ra);
  const float2* pa = a.spec + ((size_t)slot * H + 2 * pair) * Wh;
  with_radix<kColTo32>(ra, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    if (t >= rb) return;
    float2 u[R];
    load_full_bins<R>(u, pa, pa + Wh, W, t, rb);
    DftP<R, true>::run(u);
    float2* dst = sm + t * odd_pitch(R);
#pragma unroll
    for (int r = 0; r < R; ++r) dst[r] = u[r];
  });
  __syncwarp();
  PairStat ps;
  with_radix<kColTo32>(rb, [&](auto rc) {
    constexpr int R = decltype(rc)::value;
    if (t >= ra) return;
    float2 v[R];
    const int step = odd_pitch(ra);
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = sm[t + r * step];
    plan_twiddles<R, true>(v, t, ra, a.prow.tab + a.prow.tw_fwd);
    DftP<R, true>::run(v);
    if (c_out) {
      float* oa = c_out + (size_t)(2 * pair) * W;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        oa[t + r * ra] = v[r].x;
        oa[W + t + r * ra] = v[r].y;
      }
      return;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) ps.add(t + r * ra, r, v[r]);
  });
  if (c_out) return;
  const RowRed red = ps.reduce();
  if (t == 0) row_stats_final(&red, 1, a.stats + (size_t)slot * H + 2 * pair);
}

// ---------------------------------------------------------------- three stages

// f(R as a compile-time constant), the radices of the three-stage plans
template <class F>
__device__ __forceinline__ void with_radix3(int R, F&& f) {
  switch (R) {
    case 5: f(RadixC<5>{}); break;
    case 8: f(RadixC<8>{}); break;
    case 9: f(RadixC<9>{}); break;
    case 10: f(RadixC<10>{}); break;
    case 12: f(RadixC<12>{}); break;
    case 15: f(RadixC<15>{}); break;
    case 16: f(RadixC<16>{}); break;
    case 18: f(RadixC<18>{}); break;
    case 20: f(RadixC<20>{}); break;
    default: f(RadixC<25>{}); break;
  }
}

// Element q R1 R2 + k (k < R1 R2) of the order between the second and the third
// stage lies at q L + k.  L = R1 modulo 16: 16 lanes of a store, whose
// butterflies are runs of R1 consecutive elements R1 R2 apart, then meet 16
// consecutive 8-byte banks.
__host__ __device__ constexpr int row3_pitch(int r1, int r2) { return r1 * r2 + ((r1 - r1 * r2) & 15); }
__host__ __device__ inline int row3_points(const int r[3]) {
  const int a = r[1] * r[2] * odd_pitch(r[0]), b = r[2] * row3_pitch(r[0], r[1]);
  return a > b ? a : b;
}
constexpr int kRow3MaxThreads = 416;
// 64 registers (at 72, 13.8 against 12.0 us at 1440 x 2560's row forward), two radices spill a little
constexpr int kRow3Bound = 512;
__host__ __device__ inline int row3_threads(const int r[3]) {   // r[0] is the smallest
  return (r[1] * r[2] + 31) & ~31;
}

// The stages of a row pair in sm, whose barriers every thread of the block meets:
//   first  : butterfly t < R2 R3 of x[t + r R2 R3]; writes t LA + r (LA = R1 or
//            R1 + 1, odd)
//   second : butterfly t < R1 R3, t = q R1 + k: reads q LA + k + r R3 LA, twiddle
//            w_(R1 R2)^(rk); writes q L + k + r R1
//   third  : butterfly t < R1 R2: reads t + r L, twiddle w_W^(rt); its outputs
//            are t + r R1 R2
template <bool INV>
struct Row3 {
  const PassArgs& a;
  float2* sm;
  int t;
  template <class Ld>
  __device__ __forceinline__ void first(Ld&& ld) const {   // ld's reads of sm end before the writes
    with_radix3(a.prow.r3[0], [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int nb = a.prow.r3[1] * a.prow.r3[2];
      float2 u[R];
      if (t < nb) ld(u, nb);
      if (!INV) __syncthreads();
      if (t < nb) {
        DftP<R, INV>::run(u);
        float2* dst = sm + t * odd_pitch(R);
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r] = u[r];
      }
    });
    __syncthreads();
  }
  __device__ __forceinline__ void second() const {
    with_radix3(a.prow.r3[1], [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int r1 = a.prow.r3[0], r3 = a.prow.r3[2], la = odd_pitch(r1);
      const int q = (int)__umulhi((unsigned)t, a.prow.inv3), k = t - q * r1;
      float2 u[R];
      if (t < r1 * r3) {
        const float2* src = sm + q * la + k;
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = src[r * r3 * la];
      }
      __syncthreads();
      if (t < r1 * r3) {
        plan_twiddles<R, INV>(u, k, r1, a.prow.tab + a.prow.w3[0]);
        DftP<R, INV>::run(u);
        float2* dst = sm + q * row3_pitch(r1, R) + k;
#pragma unroll
        for (int r = 0; r < R; ++r) dst[r * r1] = u[r];
      }
    });
    __syncthreads();
  }
  // st(x of output 0, step, outputs), after every thread's reads where SYNC
  template <bool SYNC, class St>
  __device__ __forceinline__ void third(St&& st) const {
    with_radix3(a.prow.r3[2], [&](auto rc) {
      constexpr int R = decltype(rc)::value;
      const int nb = a.prow.r3[0] * a.prow.r3[1], L = row3_pitch(a.prow.r3[0], a.prow.r3[1]);
      float2 u[R];
      if (t < nb) {
#pragma unroll
        for (int r = 0; r < R; ++r) u[r] = sm[t + r * L];
        plan_twiddles<R, INV>(u, t, nb, a.prow.tab + a.prow.w3[1]);
        DftP<R, INV>::run(u);
      }
      if (SYNC) __syncthreads();
      if (t < nb) st(u, t, nb);
    });
  }
};

// As k_row_forward2, a row pair a block of row3_threads threads.
template <int DT>
__global__ void __launch_bounds__(kRow3Bound, 2)
    k_row_forward3(PassArgs a, const float* __restrict__ mean_sub, int warp, float2* __restrict__ out_override) {
  extern __shared__ float2 smem[];
  const int t = threadIdx.x, y0 = 2 * blockIdx.x, slot = blockIdx.y, Wh = a.W >> 1;
  load_row_pair<DT>(a, slot, y0, mean_sub, warp, t, blockDim.x, smem);
  __syncthreads();
  const Row3<false> w{a, smem, t};
  w.first([&](auto& u, int nb) {
#pragma unroll
    for (int r = 0; r < (int)(sizeof(u) / sizeof(u[0])); ++r) u[r] = smem[t + r * nb];
  });
  w.second();
  w.template third<true>([&](auto& u, int x, int step) {
#pragma unroll
    for (int r = 0; r < (int)(sizeof(u) / sizeof(u[0])); ++r) smem[x + r * step] = u[r];
  });
  __syncthreads();
  store_half_spectra(smem, (out_override ? out_override : a.spec + (size_t)slot * a.H * Wh) + (size_t)y0 * Wh, a.W, t,
                     blockDim.x);
}

// As k_row_inverse2, a row pair a block.
template <int MINB>
__global__ void __launch_bounds__(kRow3Bound, MINB) k_row_inverse3(PassArgs a, float* __restrict__ c_out) {
  extern __shared__ float2 smem[];
  __shared__ RowRed s_red[kRow3MaxThreads / 32];
  const int t = threadIdx.x, y0 = 2 * blockIdx.x, slot = blockIdx.y, W = a.W, Wh = W >> 1;
  const float2* pa = a.spec + ((size_t)slot * a.H + y0) * Wh;
  const Row3<true> w{a, smem, t};
  w.first([&](auto& u, int nb) { load_full_bins(u, pa, pa + Wh, W, t, nb); });
  w.second();
  PairStat ps;
  w.template third<false>([&](auto& u, int x, int step) {
    constexpr int R = (int)(sizeof(u) / sizeof(u[0]));
    if (c_out) {
      float* oa = c_out + (size_t)y0 * W;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        oa[x + r * step] = u[r].x;
        oa[W + x + r * step] = u[r].y;
      }
      return;
    }
#pragma unroll
    for (int r = 0; r < R; ++r) ps.add(x + r * step, r, u[r]);
  });
  if (c_out) return;
  const RowRed red = ps.reduce();
  if ((t & 31) == 0) s_red[t >> 5] = red;
  __syncthreads();
  if (t == 0) row_stats_final(s_red, blockDim.x >> 5, a.stats + (size_t)slot * a.H + y0);
}

}  // namespace prnu
