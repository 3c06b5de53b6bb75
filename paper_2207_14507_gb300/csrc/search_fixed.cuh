// search_fixed.cuh -- compile-time-planned kernels of the grid search for the
// frame sizes of the workloads (256x256, 1280x720, 1920x1080, 3840x2160).
//
// Same arithmetic as the generic kernels in search.cu (Stockham stages,
// radix-R DFTs in registers, the same packed half spectrum), with the plan,
// the frame size and the thread count known at compile time, so that every
// address is a per-thread base plus a constant (fft_fixed.cuh), and with
// fewer shared-memory passes:
//   row_forward_body : stage 0 of the row FFT takes its inputs straight from
//                      the bilinear warp (no shared-memory fill);
//   col_body         : (col_pass.cuh) two long stages each way in registers;
//   row_inverse_body : stage 0 rebuilds the two rows' full spectrum straight
//                      from global memory; the last stage's outputs are
//                      reduced to the row statistics from registers.
// Each body runs either as its own wave kernel (one launch per phase over a
// wave of candidates) or inside k_persist, one launch that schedules all
// phases of all candidates of a call as tasks (see below).
// Each frame size's kernels are instantiated in a translation unit of their
// own (search_fixed_<rows>.cu), so that they compile in parallel.
#pragma once
#include <algorithm>
#include <vector>

#include "col_pass.cuh"
#include "fft_fixed.cuh"
#include "internal.h"
#include "search_common.cuh"
#include "search_fixed.h"
#include "tma.cuh"

namespace prnu {

namespace {

// Loads of spectra: L2-only (CG) inside the persistent kernel, whose blocks
// read what other blocks of the same launch wrote into reused slots; through
// the read-only path in the wave kernels, where the spectrum was written by an
// earlier launch.
template <bool CG>
__device__ __forceinline__ float2 ld_spec(const float2* p) {
  if constexpr (CG) return __ldcg(p);
  else return __ldg(p);
}

template <int W>
__host__ __device__ constexpr size_t row_fx_smem(int ppb) {
  return (size_t)ppb * row_len2(W) * sizeof(float2) + (size_t)ppb * 32 * sizeof(WarpRed);
}
__host__ __device__ constexpr size_t col_fx_smem(int H, int nc) { return (size_t)H * nc * sizeof(float2); }

// ---------------------------------------------------------------- row forward

// The 16 warped samples x = t + r*NB0 (r < 16) of output rows y0 and y0 + 1,
// packed as one complex row (row y0 real, row y0 + 1 imaginary).  CLAMP
// false is only taken when every sample point of the row pair lies in
// [-1, W] x [-1, H], where the clamp of bilinear_pad is the identity.
template <int DT, int W, int NB0, bool CLAMP>
__device__ __forceinline__ void warp_row16(const typename StoreT<DT>::type* __restrict__ fr, int H, const WorkItem& it,
                                           float dxj, float bx0, float by0, float bx1, float by1, float2 (&v)[16]) {
#pragma unroll
  for (int r = 0; r < 16; ++r) {
    const float dx = dxj + (float)(r * NB0);
    v[r].x = bilinear_pad<DT, W, CLAMP>(fr, H, fmaf(it.a11, dx, bx0), fmaf(it.a21, dx, by0));
    v[r].y = bilinear_pad<DT, W, CLAMP>(fr, H, fmaf(it.a11, dx, bx1), fmaf(it.a21, dx, by1));
  }
}

__device__ __forceinline__ bool in_box(float qx, float qy, int W, int H) {
  return qx >= -1.f && qx <= (float)W && qy >= -1.f && qy <= (float)H;
}

// Row pairs bx*PPB .. bx*PPB+PPB-1 of candidate `is` (item slot), spectrum
// written to workspace slot `ws`.  Block = PPB groups of T threads.
template <int DT, class SP, int T, int PPB>
__device__ __forceinline__ void row_forward_body(const PassArgs& a, int is, int ws, int bx, float2* smem, int tx) {
  constexpr int W = SP::N, Wh = W / 2, L = row_len2(W);
  using S0 = Stg<SP, 0>;
  static_assert(S0::R == 16 && SP::S >= 2 && SP::S <= 3, "row plans: radix 16 first, two or three stages");
  constexpr int NB0 = S0::NB;
  const int grp = tx / T, t = tx - grp * T;
  const int H = a.H;
  const int pair = bx * PPB + grp;
  float2* A = smem + (size_t)grp * L;   // the row pair's buffer; stages 1.. run in place
  const WorkItem it = item_of(a, is);
  size_t base;
  const void* Rf = frame_of(a, it.frame, &base);
  const auto* fr = reinterpret_cast<const typename StoreT<DT>::type*>(Rf) + base;
  const int y0 = 2 * pair;
  const float cx = 0.5f * (float)(W - 1), cy = 0.5f * (float)(H - 1);
  const float dy0 = (float)y0 - cy, dy1 = dy0 + 1.f;
  const float bx0 = fmaf(it.a12, dy0, cx), by0 = fmaf(it.a22, dy0, cy);
  const float bx1 = fmaf(it.a12, dy1, cx), by1 = fmaf(it.a22, dy1, cy);
  // The sample coordinates are monotone in x, so the ends of the two rows
  // bound them all (uniform over the thread group).
  const float dxl = -cx, dxr = (float)(W - 1) - cx;
  const bool inside = in_box(fmaf(it.a11, dxl, bx0), fmaf(it.a21, dxl, by0), W, H) &&
                      in_box(fmaf(it.a11, dxr, bx0), fmaf(it.a21, dxr, by0), W, H) &&
                      in_box(fmaf(it.a11, dxl, bx1), fmaf(it.a21, dxl, by1), W, H) &&
                      in_box(fmaf(it.a11, dxr, bx1), fmaf(it.a21, dxr, by1), W, H);
  if (t < NB0) {
    float2 v[16];
    const float dxj = (float)t - cx;
    if constexpr (DT == kF32I) {
      const float *p = fr + (size_t)y0 * a.rpitch + t, *q = p + a.rpitch;
#pragma unroll
      for (int r = 0; r < 16; ++r) v[r] = make_float2(__ldg(p + r * NB0), __ldg(q + r * NB0));
    } else if (inside) warp_row16<DT, W, NB0, false>(fr, H, it, dxj, bx0, by0, bx1, by1, v);
    else warp_row16<DT, W, NB0, true>(fr, H, it, dxj, bx0, by0, bx1, by1, v);
    Dft<16, false>::run(v);
    row_store16(A, t, v);
  }
  __syncthreads();
  float2* o0 = a.spec + ((size_t)ws * H + y0) * Wh;
  float2* o1 = o0 + Wh;
  using LS = Stg<SP, SP::S - 1>;
  constexpr int R = LS::R, NS = LS::NS, LB = NS / 16 * 18;
  // Split z = G_a + i G_b into the two rows' half spectra (packed: bin 0 holds
  // (DC, Nyquist)): bin x < W/2 from z(x) and z(W - x).
  auto put = [&](int x, float2 zk, float2 zm) {
    o0[x] = make_float2(0.5f * (zk.x + zm.x), 0.5f * (zk.y - zm.y));
    o1[x] = make_float2(0.5f * (zk.y + zm.y), 0.5f * (zm.x - zk.x));
  };
  auto put0 = [&](float2 z0, float2 zn) {
    o0[0] = make_float2(z0.x, zn.x);
    o1[0] = make_float2(z0.y, zn.y);
  };
  if constexpr (SP::S == 3) {
    row_stage_ip<SP, 1, T, false>(A, t);
    __syncthreads();
  }
  // Output x = j + r*Ns of the last stage has its mirror W - x at r' = R-1-r of
  // butterfly Ns - j; j = 0 and Ns/2 are their own mirrors.
  if constexpr (R % 2 == 0 && NS % 2 == 0 && NS / 2 <= T && NS > T) {
    // a thread holds both butterflies of a mirror pair: no exchange
    if (t < NS / 2) {
      const int ja = t, jb = t == 0 ? NS / 2 : NS - t;
      float2 va[1][R], vb[1][R];
      mirror_pair_stage<R, NS, false>(A, t, va[0], vb[0]);
      if (t == 0) {
        put0(va[0][0], va[0][R / 2]);
#pragma unroll
        for (int r = 1; r < R / 2; ++r) put(r * NS, va[0][r], va[0][R - r]);
#pragma unroll
        for (int r = 0; r < R / 2; ++r) put(NS / 2 + r * NS, vb[0][r], vb[0][R - 1 - r]);
      } else {
#pragma unroll
        for (int r = 0; r < R / 2; ++r) {
          put(ja + r * NS, va[0][r], vb[0][R - 1 - r]);
          put(jb + r * NS, vb[0][r], va[0][R - 1 - r]);
        }
      }
    }
  } else if constexpr (R % 2 == 0 && NS % 2 == 0 && T % 32 == 0 && (NS / 2 + 15) / 16 * 32 <= T) {
    // one butterfly per thread, those of a mirror pair on lanes l and l ^ 16 of
    // one warp (j = 0 and Ns/2 share lane pair 0): mirror bins by shuffle
    const int p = (t >> 5) * 16 + (t & 15), h = (t >> 4) & 1;
    const int j = p == 0 ? (h ? NS / 2 : 0) : (h ? NS - p : p);
    float2 v[1][R];
    if (p < NS / 2) {
      const float2* src = A + rp2(j);
#pragma unroll
      for (int r = 0; r < R; ++r) v[0][r] = src[r * LB];
      twiddle_tab<R, NS, false, 1>(v, j);
      DftP<R, false>::run(v[0]);
    }
    float2 m[R / 2];
#pragma unroll
    for (int r = 0; r < R / 2; ++r) {
      m[r].x = __shfl_xor_sync(0xffffffffu, v[0][R - 1 - r].x, 16);
      m[r].y = __shfl_xor_sync(0xffffffffu, v[0][R - 1 - r].y, 16);
    }
    if (p < NS / 2) {
#pragma unroll
      for (int r = 0; r < R / 2; ++r) {
        if (j == 0 && r == 0) put0(v[0][0], v[0][R / 2]);
        else put(j + r * NS, v[0][r], j == 0 ? v[0][R - r] : j == NS / 2 ? v[0][R - 1 - r] : m[r]);
      }
    }
  } else if constexpr (R % 2 == 0 && NS == 16 && T == 16) {
    // one butterfly per thread of a half warp: the mirror's lane is 16 - t
    float2 v[1][R];
    const float2* src = A + rp2(t);
#pragma unroll
    for (int r = 0; r < R; ++r) v[0][r] = src[r * LB];
    twiddle_tab<R, NS, false, 1>(v, t);
    DftP<R, false>::run(v[0]);
#pragma unroll
    for (int r = 0; r < R / 2; ++r) {
      float2 m;
      m.x = __shfl_sync(0xffffffffu, v[0][R - 1 - r].x, (16 - t) & 15, 16);
      m.y = __shfl_sync(0xffffffffu, v[0][R - 1 - r].y, (16 - t) & 15, 16);
      if (t == 0 && r == 0) put0(v[0][0], v[0][R / 2]);
      else put(t + r * NS, v[0][r], t == 0 ? v[0][(R - r) % R] : m);
    }
  } else {
    // the last stage through shared memory
    row_stage_ip<SP, SP::S - 1, T, false>(A, t);
    __syncthreads();
    constexpr int MI = (Wh + T - 1) / T;
    const float2* rk = A + rp2(t);
    const float2* rm = A - t + 2 * ((-t) >> 4);   // + rp2(X) gives rp2(X - t) for X = 0 mod 16
#pragma unroll
    for (int m = 0; m < MI; ++m) {
      const int k = t + m * T;
      if (Wh % T != 0 && k >= Wh) break;
      const float2 zk = rk[m * (T / 16 * 18)];
      if (m == 0 && t == 0) put0(zk, A[rp2(Wh)]);
      else put(k, zk, rm[rp2(W - m * T)]);
    }
  }
}

// ---------------------------------------------------------------- row inverse + statistics

// Inverse row FFT of z = G_a + i G_b, the full spectrum of the packed rows
// pa and pb (W/2 bins each), by the T threads of one group (thread t) with
// buffers A and B (row layout).  Afterwards thread t < n/R_last holds the
// outputs x = t + r*Ns_last of the last stage in v (v.x row a, v.y row b).
// Holds barriers: every thread of the block calls it.
template <class SP, int T, bool CG>
__device__ __forceinline__ void row_inverse_fft(const float2* pa, const float2* pb, float2* A, int t,
                                                float2 (&v)[RowLast<SP, T>::IT][RowLast<SP, T>::R]) {
  constexpr int W = SP::N, Wh = W / 2;
  using S0 = Stg<SP, 0>;
  static_assert(S0::R == 16 && SP::S >= 2 && SP::S <= 3, "row plans: radix 16 first, two or three stages");
  constexpr int NB0 = S0::NB;   // bins j + r*NB0: r < 8 below W/2, r >= 8 mirrored
  if (t < NB0) {
    float2 u[16];
    float2 a0 = make_float2(0.f, 0.f), b0 = a0;
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      const float2 A_ = ld_spec<CG>(pa + t + r * NB0), B_ = ld_spec<CG>(pb + t + r * NB0);
      if (r == 0) {
        a0 = A_;
        b0 = B_;
      }
      u[r] = make_float2(A_.x - B_.y, A_.y + B_.x);
    }
    const float2* ma = pa + (W - t);
    const float2* mb = pb + (W - t);
#pragma unroll
    for (int r = 8; r < 16; ++r) {
      float2 A_, B_;
      if (r == 8) {   // bin W/2 - t; for t = 0 the Nyquist bin, packed in bin 0
        const int k8 = t ? Wh - t : 0;
        A_ = ld_spec<CG>(pa + k8);
        B_ = ld_spec<CG>(pb + k8);
      } else {
        A_ = ld_spec<CG>(ma - r * NB0);
        B_ = ld_spec<CG>(mb - r * NB0);
      }
      u[r] = make_float2(A_.x + B_.y, B_.x - A_.y);
    }
    if (t == 0) {   // DC and Nyquist of both rows: (re, im) = (DC, Nyquist) in bin 0
      u[0] = make_float2(a0.x, b0.x);
      u[8] = make_float2(a0.y, b0.y);
    }
    DftP<16, true>::run(u);
    row_store16(A, t, u);
  }
  __syncthreads();
  if constexpr (SP::S == 3) {
    row_stage_ip<SP, 1, T, true>(A, t);
    __syncthreads();
  }
  row_stage_last<SP, T, true>(A, t, v);
}

template <class SP, int T, int PPB, bool CG = false>
__device__ __forceinline__ void row_inverse_body(const PassArgs& a, int ws, int bx, float2* smem, int tx) {
  constexpr int W = SP::N, Wh = W / 2, L = row_len2(W);
  using GL = RowLast<SP, T>;
  static_assert(T % 16 == 0 && T * PPB % 32 == 0, "row-pair groups in half warps, whole warps in all");
  const int grp = tx / T, t = tx - grp * T;
  const int H = a.H;
  const int pair = bx * PPB + grp;
  float2* A = smem + (size_t)grp * L;
  RowRed* red = reinterpret_cast<RowRed*>(smem + (size_t)PPB * L) + grp * 32;
  const float2* pa = a.spec + ((size_t)ws * H + 2 * pair) * Wh;
  float2 v[GL::IT][GL::R];
  row_inverse_fft<SP, T, CG>(pa, pa + Wh, A, t, v);
  // per thread: max, first arg-max and energy of each row over its outputs,
  // visited in increasing x (butterfly 0's before butterfly 1's at each r), so a
  // strictly larger value is the only one that moves the arg-max: the first
  // maximum is kept without comparing indices
  float ma = -INFINITY, mb = -INFINITY;
  int ia = INT_MAX, ib = INT_MAX;
  float2 sqs[GL::IT] = {};   // a sum per butterfly: at most 16 terms
#pragma unroll
  for (int r = 0; r < GL::R; ++r) {
#pragma unroll
    for (int it = 0; it < GL::IT; ++it) {
      if (!GL::valid(t, it)) continue;
      const int x = GL::x(t, it, r);
      const float2 u = v[it][r];
      if (u.x > ma) {
        ma = u.x;
        ia = x;
      }
      if (u.y > mb) {
        mb = u.y;
        ib = x;
      }
      sqs[it] = __ffma2_rn(u, u, sqs[it]);
    }
  }
  float2 sq = sqs[0];
#pragma unroll
  for (int it = 1; it < GL::IT; ++it) sq = __fadd2_rn(sq, sqs[it]);
  // across the warp: the max by an integer reduction of the order-preserving
  // key, then the least index among the lanes that hold it (across the half
  // warp by shuffles where groups share warps); energies by an FP32 butterfly (warps are combined
  // in double by row_stats_final)
  constexpr int SEG = T % 32 == 0 ? 32 : 16;
  if constexpr (SEG == 32) {
    const int ka = __reduce_max_sync(0xffffffffu, float_key(ma));
    const int kb = __reduce_max_sync(0xffffffffu, float_key(mb));
    ia = __reduce_min_sync(0xffffffffu, float_key(ma) == ka ? ia : INT_MAX);
    ib = __reduce_min_sync(0xffffffffu, float_key(mb) == kb ? ib : INT_MAX);
    ma = key_float(ka);
    mb = key_float(kb);
  } else {
#pragma unroll
    for (int o = SEG / 2; o; o >>= 1) {
      better_f(ma, ia, __shfl_xor_sync(0xffffffffu, ma, o), __shfl_xor_sync(0xffffffffu, ia, o));
      better_f(mb, ib, __shfl_xor_sync(0xffffffffu, mb, o), __shfl_xor_sync(0xffffffffu, ib, o));
    }
  }
#pragma unroll
  for (int o = SEG / 2; o; o >>= 1) {
    sq.x += __shfl_xor_sync(0xffffffffu, sq.x, o);
    sq.y += __shfl_xor_sync(0xffffffffu, sq.y, o);
  }
  if (t % SEG == 0) red[t / SEG] = RowRed{ma, ia, mb, ib, sq.x, 0.f, sq.y, 0.f};
  __syncthreads();
  if (t == 0) row_stats_final(red, (T + SEG - 1) / SEG, a.stats + (size_t)ws * H + 2 * pair);
}

// ---------------------------------------------------------------- wave kernels

// blockIdx.y = candidate slot, or with forward units the unit u, whose row
// spectrum goes to slot a.nitems + u
template <int DT, class SP, int T, int PPB>
__device__ __forceinline__ void row_forward_block(const PassArgs& a, float2* smem) {
  const bool units = a.units || a.share > 1;
  const int u = blockIdx.y;
  if (past_count(a, u, units ? 1 : 0)) return;
  row_forward_body<DT, SP, T, PPB>(a, units ? unit_first(a, u) : u, units ? a.nitems + u : u, blockIdx.x, smem,
                                   threadIdx.x);
}
template <int DT, class SP, int T, int PPB>
__global__ void __launch_bounds__(T * PPB) k_row_forward_fx(PassArgs a) {
  extern __shared__ float4 smem4[];
  row_forward_block<DT, SP, T, PPB>(a, reinterpret_cast<float2*>(smem4));
}
// the same with registers allocated for MINB resident blocks per SM (a
// separate kernel: an explicit bound of 1 changes the allocation of the
// unbounded one)
template <int DT, class SP, int T, int PPB, int MINB>
__global__ void __launch_bounds__(T * PPB, MINB) k_row_forward_mb(PassArgs a) {
  extern __shared__ float4 smem4[];
  row_forward_block<DT, SP, T, PPB>(a, reinterpret_cast<float2*>(smem4));
}

template <class CP, int W, int NC, int MINB>
__global__ void __launch_bounds__(NC* CP::lanes, MINB) k_col_fx(PassArgs a) {
  extern __shared__ float4 smem4[];
  if (past_count(a, blockIdx.y, 0)) return;
  col_body<CP, W, NC>(a, blockIdx.y, blockIdx.y, blockIdx.x, reinterpret_cast<float2*>(smem4));
}

template <class CP, int W, int NC, int MINB, int MODE, int PFD>
__global__ void __launch_bounds__(NC* CP::lanes, MINB) k_col_tma_fx(PassArgs a, const __grid_constant__ CUtensorMap map) {
  extern __shared__ __align__(1024) float4 smem4t[];
  if (past_count(a, blockIdx.y, 0)) return;
  col_body<CP, W, NC, MODE, 0, PFD>(a, blockIdx.y, blockIdx.y, blockIdx.x, reinterpret_cast<float2*>(smem4t), &map);
}

// Forward units (see col_body PART): the forward column FFT of unit
// blockIdx.y, in place in its slot a.nitems + u; then, per candidate slot
// blockIdx.y, the product with its fingerprint and the inverse FFT from its
// unit's slot into its own.
template <class CP, int W, int NC, int MINB>
__global__ void __launch_bounds__(NC* CP::lanes, MINB) k_col_fwd_fx(PassArgs a, const __grid_constant__ CUtensorMap map) {
  extern __shared__ __align__(1024) float4 smem4f[];
  const int u = blockIdx.y;
  if (past_count(a, u, 1)) return;
  col_body<CP, W, NC, 1, 1>(a, unit_first(a, u), a.nitems + u, blockIdx.x, reinterpret_cast<float2*>(smem4f), &map);
}
template <class CP, int W, int NC, int MINB, int MODE>
__global__ void __launch_bounds__(NC* CP::lanes, MINB) k_col_inv_fx(PassArgs a, const __grid_constant__ CUtensorMap map) {
  extern __shared__ __align__(1024) float4 smem4i[];
  const int s = blockIdx.y;
  if (past_count(a, s, 0)) return;
  col_body<CP, W, NC, MODE, 2>(a, s, s, blockIdx.x, reinterpret_cast<float2*>(smem4i), &map,
                               a.nitems + unit_of_slot(a, s));
}

template <class SP, int T, int PPB>
__global__ void __launch_bounds__(T * PPB) k_row_inverse_fx(PassArgs a) {
  extern __shared__ float4 smem4[];
  if (past_count(a, blockIdx.y, 0)) return;
  row_inverse_body<SP, T, PPB>(a, blockIdx.y, blockIdx.x, reinterpret_cast<float2*>(smem4), threadIdx.x);
}
template <class SP, int T, int PPB, int MINB>
__global__ void __launch_bounds__(T * PPB, MINB) k_row_inverse_mb(PassArgs a) {
  extern __shared__ float4 smem4[];
  if (past_count(a, blockIdx.y, 0)) return;
  row_inverse_body<SP, T, PPB>(a, blockIdx.y, blockIdx.x, reinterpret_cast<float2*>(smem4), threadIdx.x);
}

// ---------------------------------------------------------------- persistent kernel

// Task bodies, inlined into k_persist.  The kernel hands them a thread index
// that the compiler cannot prove loop-invariant (see k_persist), so the
// per-thread index arithmetic of each task is computed inside its own branch
// instead of being hoisted out of the task loop, where the three tasks'
// values would all stay live at once.
template <int DT, class SP, int T, int PPB>
__device__ __forceinline__ void row_forward_task(const PassArgs& a, int is, int ws, int bx, float2* smem, int tx) {
  row_forward_body<DT, SP, T, PPB>(a, is, ws, bx, smem, tx);
}
// The column pass as a task of the persistent kernel, whose register bound
// (80 at 1080p) holds no 30-point butterfly: three radix stages, a pair of
// adjacent columns per thread, loads and stores by every thread itself, L2
// only.  The same steps as col_body (col_pass.cuh).

// The fingerprint bins (i, col0) and (i, col0 + 1) for i = j + r*NS, from the
// strip layout (col0 even: one vector).
template <int R, int NS, int H>
__device__ __forceinline__ void load_fp_pair(const FpDesc& fp, int j, int col0, float2 (&s)[2][R]) {
  const size_t b = (((size_t)(col0 >> 2) * H + j) * 4 + (col0 & 3)) / 2;
  if (fp.dtype == kF32) {
    const float4* p = reinterpret_cast<const float4*>(fp.spec) + b;
#pragma unroll
    for (int r = 0; r < R; ++r) split2(__ldg(p + r * NS * 2), s[0][r], s[1][r]);
  } else {
    const float2* p = reinterpret_cast<const float2*>(fp.spec) + b;   // two __half2
#pragma unroll
    for (int r = 0; r < R; ++r) {
      const float2 u = __ldg(p + r * NS * 2);
      s[0][r] = __half22float2(*reinterpret_cast<const __half2*>(&u.x));
      s[1][r] = __half22float2(*reinterpret_cast<const __half2*>(&u.y));
    }
  }
}
template <class SP, int W, int NC, int T>
__device__ __forceinline__ void col_task(const PassArgs& a, int is, int ws, int bx, float2* sm) {
  constexpr int H = SP::N, Wh = W / 2;
  using IS = typename SP::Rev;
  using M = ColMap<NC, T>;
  constexpr int NP = M::NP, TJ = M::TJ;
  static_assert(Wh % NC == 0, "strips tile the half spectrum");
  const int t = threadIdx.x;
  const int c0 = bx * NC;
  const int cp = t % NP, j0 = t / NP;
  const int col0 = c0 + 2 * cp;
  float2* Z = a.spec + (size_t)ws * H * Wh;
  float4* sm4 = reinterpret_cast<float4*>(sm);
  const WorkItem wi = item_of(a, is);
  const FpDesc fp = a.fps[wi.fp];
  {  // forward stage 0 from global memory
    using G = Stg<SP, 0>;
    constexpr int IT = (G::NB + TJ - 1) / TJ;
#pragma unroll
    for (int it = 0; it < IT; ++it) {
      const int j = j0 + it * TJ;
      if (G::NB % TJ != 0 && j >= G::NB) continue;
      float2 v[2][G::R];
      const float4* src = reinterpret_cast<const float4*>(Z + (size_t)j * Wh + col0);
#pragma unroll
      for (int r = 0; r < G::R; ++r) split2(__ldcg(src + (size_t)r * G::NB * (Wh / 2)), v[0][r], v[1][r]);
      Dft<G::R, false>::run(v[0]);
      Dft<G::R, false>::run(v[1]);
      float4* dst = sm4 + j * G::R * NP + cp;
#pragma unroll
      for (int r = 0; r < G::R; ++r) dst[r * NP] = join2(v[0][r], v[1][r]);
    }
  }
  __syncthreads();
  ColStages<SP, 1, SP::S - 1, T, NC, false>::run(sm4, t);
  // last forward stage -> spectrum product -> first inverse stage, in registers
  using FL = Stg<SP, SP::S - 1>;
  using I0 = Stg<IS, 0>;
  static_assert(I0::R == FL::R && I0::NB == FL::NB && FL::NB == FL::NS, "register hand-off needs the reversed plan");
  constexpr int IT = (FL::NB + TJ - 1) / TJ;
  float2 v[IT][2][FL::R];
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int j = j0 + it * TJ;
    if (FL::NB % TJ != 0 && j >= FL::NB) continue;
    const float4* src = sm4 + j * NP + cp;
#pragma unroll
    for (int r = 0; r < FL::R; ++r) split2(src[r * FL::NB * NP], v[it][0][r], v[it][1][r]);
  }
  __syncthreads();
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int j = j0 + it * TJ;
    if (FL::NB % TJ != 0 && j >= FL::NB) continue;
    twiddle_tab<FL::R, FL::NS, false, 2>(v[it], j);
    Dft<FL::R, false>::run(v[it][0]);
    Dft<FL::R, false>::run(v[it][1]);
  }
  // thread holds bins i = j + r*NS of columns col0 and col0 + 1
  if (c0 == 0) {
    // packed column 0 (DC + i*Nyquist): the product needs bin H - i as well
    if (cp == 0) {
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const int j = j0 + it * TJ;
        if (FL::NB % TJ != 0 && j >= FL::NB) continue;
#pragma unroll
        for (int r = 0; r < FL::R; ++r) sm[j + r * FL::NS] = v[it][0][r];
      }
    }
    __syncthreads();
    if (cp == 0) {
#pragma unroll
      for (int it = 0; it < IT; ++it) {
        const int j = j0 + it * TJ;
        if (FL::NB % TJ != 0 && j >= FL::NB) continue;
#pragma unroll
        for (int r = 0; r < FL::R; ++r) {
          const int i = j + r * FL::NS;
          const int im = i == 0 ? 0 : H - i;
          v[it][0][r] = packed_col0_product(v[it][0][r], sm[im], load_fp(fp, i, 0, H, Wh), load_fp(fp, im, 0, H, Wh));
        }
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int it = 0; it < IT; ++it) {
    const int j = j0 + it * TJ;
    if (FL::NB % TJ != 0 && j >= FL::NB) continue;
    float2 sf[2][FL::R];
    load_fp_pair<FL::R, FL::NS, H>(fp, j, col0, sf);
#pragma unroll
    for (int r = 0; r < FL::R; ++r) {
      if (col0 != 0) v[it][0][r] = c_conj_mul(v[it][0][r], sf[0][r]);
      v[it][1][r] = c_conj_mul(v[it][1][r], sf[1][r]);
    }
    Dft<FL::R, true>::run(v[it][0]);
    Dft<FL::R, true>::run(v[it][1]);
    float4* dst = sm4 + j * FL::R * NP + cp;
#pragma unroll
    for (int r = 0; r < FL::R; ++r) dst[r * NP] = join2(v[it][0][r], v[it][1][r]);
  }
  __syncthreads();
  ColStages<IS, 1, IS::S - 1, T, NC, true>::run(sm4, t);
  {  // last inverse stage: shared memory -> global memory
    using G = Stg<IS, IS::S - 1>;
    static_assert(G::NB == G::NS, "last stage");
    constexpr int ITL = (G::NB + TJ - 1) / TJ;
#pragma unroll
    for (int it = 0; it < ITL; ++it) {
      const int j = j0 + it * TJ;
      if (G::NB % TJ != 0 && j >= G::NB) continue;
      float2 w[2][G::R];
      const float4* src = sm4 + j * NP + cp;
#pragma unroll
      for (int r = 0; r < G::R; ++r) split2(src[r * G::NB * NP], w[0][r], w[1][r]);
      twiddle_tab<G::R, G::NS, true, 2>(w, j);
      Dft<G::R, true>::run(w[0]);
      Dft<G::R, true>::run(w[1]);
      float4* dst = reinterpret_cast<float4*>(Z + (size_t)j * Wh + col0);
#pragma unroll
      for (int r = 0; r < G::R; ++r) dst[(size_t)r * G::NS * (Wh / 2)] = join2(w[0][r], w[1][r]);
    }
  }
}
template <class SP, int T, int PPB>
__device__ __forceinline__ void row_inverse_task(const PassArgs& a, int ws, int bx, float2* smem, int tx) {
  row_inverse_body<SP, T, PPB, true>(a, ws, bx, smem, tx);
}

// The energy of window pair `p` outside the window's columns (and of its rows
// inside the window only), this thread's part; the rows by the planned inverse
// row FFT of the T threads of a group (thread t) in its buffer A.
template <class SP, int T>
__device__ __forceinline__ double window_pair_energy(const PassArgs& a, const float2* Z, const FinPeak& pk, int p, int t,
                                                     float2* A) {
  constexpr int W = SP::N, Wh = W / 2;
  using SL = RowLast<SP, T>;
  const float2* pa = Z + (size_t)(2 * p) * Wh;
  float2 V[SL::IT][SL::R];
  row_inverse_fft<SP, T, true>(pa, pa + Wh, A, t, V);
  PairEnergy e;
#pragma unroll
  for (int it = 0; it < SL::IT; ++it) {
    if (!SL::valid(t, it)) break;
#pragma unroll
    for (int r = 0; r < SL::R; ++r) {
      const int x = SL::x(t, it, r);
      if (cdist(x, pk.px, W) > kHalfWindow) e.add(V[it][r]);
    }
  }
  return e.total(cdist(2 * p, pk.py, a.H) <= kHalfWindow, cdist(2 * p + 1, pk.py, a.H) <= kHalfWindow);
}

// One candidate by PPB groups of T threads: group g takes row shares and window
// pairs g, g + PPB, ..
template <class SP, int T, int PPB>
__device__ __forceinline__ void finalize_task(const PassArgs& a, int is, int ws, float2* smem, int tx) {
  constexpr int W = SP::N, Wh = W / 2, L = row_len2(W), TB = T * PPB;
  static_assert(T % 32 == 0, "groups of whole warps: their shares end in warp reductions");
  __shared__ double red[kFinParts][T / 32];
  const int t = tx, grp = t / T, tg = t - grp * T;
  const RowStat* st = a.stats + (size_t)ws * a.H;
  const float2* Z = a.spec + (size_t)ws * a.H * Wh;
  const FinPeak pk = block_peak(st, a.H, W, t, TB, reinterpret_cast<WarpRed*>(smem + (size_t)PPB * L));
  for (int q = grp; q < kFinRowParts; q += PPB) part_warp(row_share(st, a.H, pk.py, q, tg, T), tg, red[q]);
#pragma unroll 1
  for (int b0 = 0; b0 < kFinPairParts; b0 += PPB) {
    const int b = b0 + grp;
    const double e = window_pair_energy<SP, T>(a, Z, pk, window_pair(pk.py, b % kFinPairParts, a.H), tg,
                                               smem + (size_t)grp * L);
    if (b < kFinPairParts) part_warp(e, tg, red[kFinRowParts + b]);
    __syncthreads();   // the row buffers are free again
  }
  if (t == 0) {
    double parts[kFinParts];
#pragma unroll
    for (int k = 0; k < kFinParts; ++k) parts[k] = part_total(red[k], T / 32);
    finish_candidate(a, is, pk, parts);
  }
}
// One block per candidate of the wave, PPB row pairs of the window at a time.
template <class SP, int T, int PPB>
__global__ void __launch_bounds__(T * PPB) k_finalize_fx(PassArgs a) {
  if (past_count(a, blockIdx.x, 0)) return;
  extern __shared__ float4 smem4[];
  finalize_task<SP, T, PPB>(a, blockIdx.x, blockIdx.x, reinterpret_cast<float2*>(smem4), threadIdx.x);
}
// One block per window pair (blockIdx.y) of a candidate; k_finalize_sum ends it.
template <class SP, int T>
__global__ void __launch_bounds__(T) k_finalize_part_fx(PassArgs a) {
  if (past_count(a, blockIdx.x, 0)) return;
  extern __shared__ float4 smem4[];
  __shared__ double red[2][T / 32];
  constexpr int W = SP::N, Wh = W / 2, L = row_len2(W);
  float2* smem = reinterpret_cast<float2*>(smem4);
  const int s = blockIdx.x, b = blockIdx.y, t = threadIdx.x;
  const RowStat* st = a.stats + (size_t)s * a.H;
  const FinPeak pk = block_peak(st, a.H, W, t, T, reinterpret_cast<WarpRed*>(smem + L));
  if (b < kFinRowParts) part_warp(row_share(st, a.H, pk.py, b, t, T), t, red[0]);
  part_warp(window_pair_energy<SP, T>(a, a.spec + (size_t)s * a.H * Wh, pk, window_pair(pk.py, b, a.H), t, smem), t,
            red[1]);
  __syncthreads();
  if (t == 0) {
    double* parts = fin_scratch(a, s, pk.py);
    if (b < kFinRowParts) parts[b] = part_total(red[0], T / 32);
    parts[kFinRowParts + b] = part_total(red[1], T / 32);
  }
  if (b == 0 && t == 0) park_peak(a, s, pk);
}

//
// One launch runs every phase of every candidate of a call.  Blocks take
// tasks by an atomic ticket.  Ticket order is a skewed pipeline: step s holds
// the row-forward tasks of candidate s, the column tasks of s-1, the
// row-inverse tasks of s-2 and the finalisation of s-3, so each task depends
// only on tasks with smaller tickets, which running blocks hold: the kernel
// cannot deadlock, whatever number of blocks is resident.  A task waits
// (bounded, with back-off) for the per-candidate count of its inputs; on
// timeout it raises the error flag and gives up instead of hanging.  Spectra
// and row statistics live in S workspace slots used round-robin (candidate g
// in slot g % S), so only about four candidates' spectra are in flight and
// they stay in L2; a row-forward task also waits for the finalisation of
// candidate g - S, the previous user of its slot.

constexpr long long kSpinLimit = 1ll << 23;   // ~2 s with the back-off below

__device__ __forceinline__ bool wait_count(const int* c, int need, int* err) {
  for (long long it = 0; it < kSpinLimit; ++it) {
    if (*(volatile const int*)c >= need) {
      __threadfence();
      return true;
    }
    if (*(volatile int*)err) return false;
    __nanosleep(it < 32 ? 64 : 256);
  }
  atomicExch(err, 1);
  return false;
}

template <int DT, class RS, int RT, int PPB, class CS, int NC>
__global__ void __launch_bounds__(RT * PPB, RT * PPB <= 384 ? 2 : 1)
    k_persist(const __grid_constant__ PassArgs a, const __grid_constant__ PersistArgs p) {
  constexpr int TB = RT * PPB;
  extern __shared__ float2 smem[];
  __shared__ int s_tk[2], s_ok, s_zero;
  static_assert(RT * PPB >= 64, "warp 1 publishes completions");
  const int H = a.H, Wh = a.W / 2;
  const int NRF = (H / 2) / PPB;
  const int NCOL = (Wh + NC - 1) / NC;
  const int NRI = NRF;
  const int TPS = NRF + NCOL + NRI + 1;
  const int total = (p.G + 3) * TPS;
  if (threadIdx.x == 0) {
    s_tk[0] = atomicAdd(p.ticket, 1);
    s_zero = 0;
  }
  __syncthreads();
  for (int iter = 0;; ++iter) {
    const int tk = s_tk[iter & 1];
    if (tk >= total) break;
    // the next ticket is fetched now and used after this task: its latency
    // overlaps the task instead of stalling the block
    int nxt = 0;
    if (threadIdx.x == 0) nxt = atomicAdd(p.ticket, 1);
    const int step = tk / TPS, r = tk - (tk / TPS) * TPS;
    int type, g, idx;
    if (r < NRF) {
      type = 0; g = step; idx = r;
    } else if (r < NRF + NCOL) {
      type = 1; g = step - 1; idx = r - NRF;
    } else if (r < NRF + NCOL + NRI) {
      type = 2; g = step - 2; idx = r - NRF - NCOL;
    } else {
      type = 3; g = step - 3; idx = 0;
    }
    if (g >= 0 && g < p.G) {   // uniform over the block
      const int ws = g % p.S;
      if (threadIdx.x == 0) {
        const int* dep = nullptr;
        int need = 1;
        if (type == 0) {
          if (g >= p.S) dep = p.fin_done + (g - p.S);
        } else if (type == 1) {
          dep = p.rf_done + g;
          need = NRF;
        } else if (type == 2) {
          dep = p.col_done + g;
          need = NCOL;
        } else {
          dep = p.ri_done + g;
          need = NRI;
        }
        s_ok = dep ? wait_count(dep, need + a.stall, p.error) : 1;   // the test hook waits for one count too many
      }
      __syncthreads();
      const bool ok = s_ok;
      if (ok) {
        const int tx = threadIdx.x + *(volatile int*)&s_zero;   // == threadIdx.x
        if (type == 0) row_forward_task<DT, RS, RT, PPB>(a, g, ws, idx, smem, tx);
        else if (type == 1) col_task<CS, RS::N, NC, TB>(a, g, ws, idx, smem);
        else if (type == 2) row_inverse_task<RS, RT, PPB>(a, ws, idx, smem, tx);
        else finalize_task<RS, RT, PPB>(a, g, ws, smem, tx);
      }
      __syncthreads();
      // completion is published by warp 1, so that warp 0 can go on to the
      // next ticket's dependency while the fence drains
      if (threadIdx.x == 32 && ok) {
        __threadfence();
        int* c = type == 0 ? p.rf_done : type == 1 ? p.col_done : type == 2 ? p.ri_done : p.fin_done;
        atomicAdd(c + g, 1);
      }
    }
    if (threadIdx.x == 0) s_tk[(iter + 1) & 1] = nxt;
    __syncthreads();
  }
}

// ---------------------------------------------------------------- registry

// row pairs of the 11-row window recomputed at once by the finalisation
constexpr int kFinPairs = 3;

// RT threads per row pair in the row forward kernel, RTI in the row inverse
// (and in the finalisation); CP the column pass's plan, CS the three-stage
// plan of the persistent kernel's column task
template <class RS, int RT, class CP, class CS, int RTI = RT>
struct ShapeDef {
  static constexpr int W = RS::N, H = CP::H;
  static constexpr int FT = (RTI + 31) / 32 * 32;   // of a row pair in the finalisation: whole warps
  static_assert(CS::N == H, "column plans of one length");
  // NC columns per block, at least MINB resident blocks per SM
  // MODE: 0 plain loads and stores, 1 strip by TMA, 2 strip by TMA and fingerprint by bulk copies
  static FixedCol col_entry(void* fn, int nc, int mode) {
    allow_max_dynamic_smem(fn);
    return FixedCol{nc, nc * CP::lanes, col_pass_smem<CP>(nc, mode), fn, mode != 0, tma_box_rows(H, nc), mode};
  }
  template <int NC, int MINB, int MODE, int PFD = 0>
  static FixedCol col() {
    if constexpr (MODE > 0) return col_entry((void*)k_col_tma_fx<CP, W, NC, MINB, MODE, PFD>, NC, MODE);
    else return col_entry((void*)k_col_fx<CP, W, NC, MINB>, NC, MODE);
  }
  // the split column pass of forward units (NC columns, MINB blocks)
  template <int NC, int MINB>
  static FixedCol col_fwd() {
    return col_entry((void*)k_col_fwd_fx<CP, W, NC, MINB>, NC, 1);
  }
  template <int NC, int MINB, int MODE>
  static FixedCol col_inv() {
    return col_entry((void*)k_col_inv_fx<CP, W, NC, MINB, MODE>, NC, MODE);
  }
  // RIMB, RFMB: resident row-inverse and row-forward blocks per SM to allocate
  // registers for (0: no bound)
  template <int DT, int PPB, int RFMB>
  static void* row_fwd() {
    void* f;
    if constexpr (RFMB > 0) f = (void*)k_row_forward_mb<DT, RS, RT, PPB, RFMB>;
    else f = (void*)k_row_forward_fx<DT, RS, RT, PPB>;
    allow_max_dynamic_smem(f);
    return f;
  }
  template <int PPB, int RIMB = 0, int RFMB = 0>
  static FixedRow row() {
    FixedRow r{};
    r.ppb = PPB;
    r.threads = RT;
    r.threads_inv = RTI;
    r.smem = row_fx_smem<W>(PPB);
    r.fwd[kF32] = row_fwd<kF32, PPB, RFMB>();
    r.fwd[kF16] = row_fwd<kF16, PPB, RFMB>();
    r.fwd[kBF16] = row_fwd<kBF16, PPB, RFMB>();
    r.fwd[kF16P] = row_fwd<kF16P, PPB, RFMB>();
    r.fwd[kBF16P] = row_fwd<kBF16P, PPB, RFMB>();
    r.fwd[kF32I] = row_fwd<kF32I, PPB, RFMB>();
    if constexpr (RIMB > 0) r.inv = (void*)k_row_inverse_mb<RS, RTI, PPB, RIMB>;
    else r.inv = (void*)k_row_inverse_fx<RS, RTI, PPB>;
    // A block per window pair where a pair's FFT fills one (us per 1000
    // candidates, one block per candidate first: 1080p 124 -> 69, 4K 258 -> 157,
    // 720p 112 -> 61; 256, one warp a pair: 35 -> 38)
    r.fin_split = FT > 32;
    r.fin_threads = r.fin_split ? FT : FT * kFinPairs;
    r.fin_smem = row_fx_smem<W>(r.fin_split ? 1 : kFinPairs);
    if constexpr (FT > 32) r.fin = (void*)k_finalize_part_fx<RS, FT>;
    else r.fin = (void*)k_finalize_fx<RS, FT, kFinPairs>;
    allow_max_dynamic_smem(r.fin);
    allow_max_dynamic_smem(r.inv);
    return r;
  }
  // PRT threads per row pair (PRT * PPB per block, also the column task's
  // threads): chosen so that every stage holds one butterfly per thread
  template <int PRT, int PPB, int NC, class PRS = RS>
  static FixedPersist persist() {
    FixedPersist f{};
    f.ppb = PPB;
    f.nc = NC;
    f.threads = PRT * PPB;
    const size_t rs = row_fx_smem<W>(PPB);
    const size_t cs = col_fx_smem(H, NC);
    const size_t fs = row_fx_smem<W>(PPB);
    f.smem = std::max(rs, std::max(cs, fs));
    f.fn[kF32] = (void*)k_persist<kF32, PRS, PRT, PPB, CS, NC>;
    f.fn[kF16] = (void*)k_persist<kF16, PRS, PRT, PPB, CS, NC>;
    f.fn[kBF16] = (void*)k_persist<kBF16, PRS, PRT, PPB, CS, NC>;
    for (int d = 0; d < 3; ++d) {
      allow_max_dynamic_smem(f.fn[d]);
      int nb = 0;
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, f.fn[d], f.threads, f.smem);
      f.blocks_per_sm[d] = std::max(1, nb);
    }
    return f;
  }
  // split: the forward half, the inverse half and, optionally, the one for FP16
  // fingerprints only (mode 4)
  static FixedShape make(std::vector<FixedRow> rows, std::vector<FixedCol> cols, std::vector<FixedCol> split,
                         FixedPersist ps) {
    FixedShape s{};
    s.W = W;
    s.H = H;
    s.rows = std::move(rows);
    s.cols = std::move(cols);
    s.col_fwd = split.at(0);
    s.col_inv = split.at(1);
    if (split.size() > 2) s.col_inv_h = split[2];
    s.persist = ps;
    return s;
  }
};

}  // namespace

}  // namespace prnu
