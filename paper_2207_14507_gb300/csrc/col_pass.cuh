// col_pass.cuh -- the column pass of the compile-time-planned kernels: forward
// column FFT, product with the fingerprint's spectrum, inverse column FFT of a
// strip of NC columns of one candidate's packed half spectrum.
//
// The transform of H = RA * RB points takes two stages each way, one thread
// per column and butterfly, a whole radix-RA or radix-RB butterfly in its
// registers (30 to 48 points): the strip crosses shared memory 6 times (plus
// the fingerprint's once) where three stages with two columns per thread
// crossed it 10 times.  Those were bound by the L1 data pipe
// (67% of its peak, a quarter of it bank conflicts and spilled registers) and
// by the barriers between its stages.  At 1080p FP32 (ncu, 64 candidates):
// 3.5 M -> 2.3 M warp instructions a candidate, L1 data pipe 67% -> 49%, L1 hit
// rate of the twiddles 49% -> 99%, 5.38 -> 4.25 us a candidate; with the
// fingerprint in contiguous strips (load_fp_strips) 3.72.  What bounds it
// now is the movement of the strip, two TMA copies in rows of 32 bytes (with the
// fingerprint's a third, movement alone took 3.35 of 4.18 us), and latency: 13.5 to 18
// warps per SM (registers and the strips' shared memory), no other unit above 50%.  Each size's variants and
// their times stand at its registry entry (search_fixed_<rows>.cu).
//
//   stage A : butterfly j < RB reads x[j + r RB], r < RA; writes j RA + r
//   stage B : butterfly j < RA reads x[j + r RA], r < RB, twiddle w_H^(rj);
//             leaves bins j + r RA in its registers
//   product : with the fingerprint's bins j + r RA
//   inverse stage B: the same thread's bins; writes j RB + r
//   inverse stage A: butterfly j < RB reads x[j + r RB], twiddle w_H^(-rj);
//             leaves rows j + r RB
//
// Between two stages the strip lies in rows of NC elements in groups of RA
// (RB) rows at an odd pitch LA (LB), so that the threads of a warp, which hold
// consecutive j and columns, store to distinct banks; TMA's side of the strip
// is dense.  Every shared address is a per-thread base plus a constant.
#pragma once
#include "col_generic.cuh"
#include "common.cuh"
#include "fft_fixed.cuh"
#include "fft_packed.cuh"
#include "search_common.cuh"
#include "search_fixed.h"
#include "tma.cuh"

namespace prnu {

namespace {

template <int H_, int RA_, int RB_>
struct ColPlan {
  static constexpr int H = H_, RA = RA_, RB = RB_;
  static constexpr int LA = RA | 1, LB = RB | 1;
  static constexpr int rows = RB * LA > RA * LB ? RB * LA : RA * LB;   // of the strip buffer
  static constexpr int lanes = RA > RB ? RA : RB;                      // threads per column
  static_assert(RA * RB == H, "two radices");
};

// bytes per fingerprint bin of the separate fingerprint region (MODE 3: FP32
// or FP16 bins; MODE 4: FP16 bins only)
__host__ __device__ constexpr int fp_region_bin(int mode) { return mode == 3 ? 8 : mode == 4 ? 4 : 0; }
// the strip buffer, 128-byte aligned; then MODE 2: the two packed column-0
// scratch columns, MODE 3 and 4: the fingerprint strip
template <class CP>
__host__ __device__ constexpr size_t col_buf_bytes(int nc) {
  return ((size_t)CP::rows * nc * sizeof(float2) + 127) / 128 * 128;
}
// The fingerprint's strips of 4 columns lie one after the other in shared
// memory, this many bytes apart beyond their own, so that the columns a warp
// reads together fall in distinct banks.
__host__ __device__ constexpr int fp_strip_pad(int nc) { return nc > 4 ? 512 / nc : 0; }
__host__ __device__ constexpr size_t fp_strips_bytes(int H, int nc, int es) {
  return (size_t)(nc / 4) * ((size_t)H * 4 * es + fp_strip_pad(nc));
}
template <class CP>
__host__ __device__ constexpr size_t col_pass_smem(int nc, int mode) {
  return col_buf_bytes<CP>(nc) + (mode == 2  ? 2 * (size_t)CP::H * sizeof(float2)
                                  : mode > 2 ? fp_strips_bytes(CP::H, nc, fp_region_bin(mode))
                                             : 0);
}
constexpr long long kTmaWaitPolls = 1ll << 20;   // polls of mbarrier.try_wait before giving up

// Every thread of the block: wait for phase `ph` of `bar`; on a wait that
// runs out anywhere the error flag goes up, the copies get one more bounded
// wait to land (and those of bar2), and false comes back to all.  Holds a
// barrier.
__device__ __forceinline__ bool block_wait(uint64_t* bar, uint32_t ph, int* err, uint64_t* bar2 = nullptr) {
  const bool ok = mbar_wait_bounded(bar, ph, kTmaWaitPolls);
  if (__syncthreads_or(!ok)) {
    if (threadIdx.x == 0) {
      if (err) atomicExch(err, 1);
      mbar_wait_bounded(bar, ph, kTmaWaitPolls);
      if (bar2) mbar_wait_bounded(bar2, 0, kTmaWaitPolls);
    }
    __syncthreads();
    return false;
  }
  return true;
}

// the fingerprint's NC columns from c0 to shared memory at dst, completing on
// bar: a contiguous copy per strip of 4 (the spectrum's own strips come as rows
// of 32 bytes, of which a TMA unit moves one in about 1.4 cycles: the
// fingerprint's, copied that way too, took a sixth of the pass)
template <int H, int NC>
__device__ __forceinline__ void load_fp_strips(const FpDesc& fp, int c0, char* dst, uint64_t* bar) {
  const uint32_t bytes = H * 4 * (fp.dtype == kF32 ? 8 : 4);
  const char* src = static_cast<const char*>(fp.spec) + (size_t)(c0 / 4) * bytes;
  mbar_expect_tx(bar, NC / 4 * bytes);
#pragma unroll 1
  for (int q = 0; q < NC / 4; ++q) bulk_load(dst + q * (bytes + fp_strip_pad(NC)), src + q * bytes, bytes, bar);
}

// Columns bx*NC .. bx*NC+NC-1 of candidate `is` in workspace slot `ws`, by
// T >= NC * CP::lanes threads.
// MODE 0: every thread loads and stores its own elements.  MODE >= 1: the
// strip comes into shared memory by TMA tile copies through `map` (the
// workspace spectra as a [slots*H][W] float tensor) and leaves the same way.
// MODE 2: the fingerprint's strips come by bulk copies, into the strip buffer once
// stage B has taken its inputs (the packed column-0 scratch then sits after
// the buffer).  MODE 3 and 4: they come into their own
// region after the strip buffer, copied from the start together with the
// strip (MODE 4 sizes the region for FP16 bins and takes FP16 fingerprints
// only).  A TMA wait that runs out raises a.err and abandons the
// candidate.
// PART splits the pass for forward units (candidates that share a frame and
// a grid node): PART 1 runs the forward column FFT only and stores its
// output, in natural order, back to slot ws; PART 2 loads that output from
// slot src_ws and runs the product and the inverse FFT into slot ws.  PART 1
// then PART 2 compute bit for bit what PART 0 (the whole pass) computes.
// PART 1 and 2 need TMA (MODE >= 1); PART 2 takes MODE >= 2.
// PFD > 0: each block also asks for the strip PFD strips on (of the wave's
// slots) to be brought into L2; PART 0 only.
template <class CP, int W, int NC, int MODE = 0, int PART = 0, int PFD = 0>
__device__ __forceinline__ void col_body(const PassArgs& a, int is, int ws, int bx, float2* sm,
                                         const CUtensorMap* map = nullptr, int src_ws = -1) {
  constexpr bool TMA = MODE >= 1, FPT = MODE >= 2 && PART != 1, FPSEP = MODE >= 3 && PART != 1;
  static_assert(PFD == 0 || (TMA && PART == 0), "prefetches go with the whole pass by TMA");
  static_assert(PART == 0 || TMA, "the split column pass moves its strips by TMA");
  constexpr int H = CP::H, Wh = W / 2, RA = CP::RA, RB = CP::RB, LA = CP::LA, LB = CP::LB;
  static_assert(Wh % NC == 0, "strips tile the half spectrum");
  if (src_ws < 0) src_ws = ws;
  const int t = threadIdx.x, c = t % NC, j = t / NC;
  const bool act_a = j < RB, act_b = j < RA;
  const int c0 = bx * NC, col = c0 + c;
  const WorkItem wi = item_of(a, is);
  const FpDesc fp = a.fps[wi.fp];
  if constexpr (MODE == 4 && PART != 1) {
    // an FP32 strip is twice the region: whoever launched this variant for it
    // (launch_fixed_wave takes another) gets an error, not the memory behind
    if (fp.dtype == kF32) {
      if (threadIdx.x == 0 && a.err) atomicExch(a.err, 1);
      return;
    }
  }
  char* const fpsm = reinterpret_cast<char*>(sm) + (FPSEP ? col_buf_bytes<CP>(NC) : 0);

  constexpr int BR = tma_box_rows(H, NC);
  __shared__ uint64_t s_bar, s_fbar;
  const bool fp32 = MODE != 4 && fp.dtype == kF32;   // MODE 4 takes FP16 fingerprints only (launch_fixed_wave)
  if constexpr (TMA) {
    static_assert(BR > 0, "no TMA box for this strip");
    if (t == 0) {
      mbar_init(&s_bar, 1);
      if (FPT) mbar_init(&s_fbar, 1);
      fence_mbar_init();
    }
    __syncthreads();
    if (t == 0) {
      mbar_expect_tx(&s_bar, H * NC * 8 + (a.stall ? 16 : 0));   // the test hook waits for bytes that never come
#pragma unroll 1
      for (int b = 0; b < H / BR; ++b) tma_load_2d(sm + b * BR * NC, map, 2 * c0, src_ws * H + b * BR, &s_bar);
      if (FPSEP) load_fp_strips<H, NC>(fp, c0, fpsm, &s_fbar);
      if constexpr (PFD > 0) {   // the strip PFD strips on, into L2
        const int n = is * (Wh / NC) + bx + PFD, s2 = n / (Wh / NC), b2 = n - s2 * (Wh / NC);
        if (s2 < a.nitems) {
#pragma unroll 1
          for (int b = 0; b < H / BR; ++b) tma_prefetch_2d(map, 2 * b2 * NC, s2 * H + b * BR);
        }
      }
    }
    if (!block_wait(&s_bar, 0, a.err, FPSEP ? &s_fbar : nullptr)) return;
  }

  float2* Z = a.spec + (size_t)ws * H * Wh;
  float2 v[1][RB];   // bins j + r RA
  if constexpr (PART != 2) {
    {
      float2 u[RA];
      if (act_a) {
        if constexpr (TMA) {
          const float2* src = sm + j * NC + c;
#pragma unroll
          for (int r = 0; r < RA; ++r) u[r] = src[r * RB * NC];
        } else {
          const float2* src = Z + (size_t)j * Wh + col;
#pragma unroll
          for (int r = 0; r < RA; ++r) u[r] = __ldg(src + (size_t)r * RB * Wh);
        }
      }
      if constexpr (TMA) __syncthreads();
      if (act_a) {
        DftP<RA, false>::run(u);
        float2* dst = sm + j * LA * NC + c;
#pragma unroll
        for (int r = 0; r < RA; ++r) dst[r * NC] = u[r];
      }
    }
    __syncthreads();
    if (act_b) {
      const float2* src = sm + j * NC + c;
#pragma unroll
      for (int r = 0; r < RB; ++r) v[0][r] = src[r * LA * NC];
    }
  } else if (act_b) {
    const float2* src = sm + j * NC + c;
#pragma unroll
    for (int r = 0; r < RB; ++r) v[0][r] = src[r * RA * NC];
  }
  if constexpr (FPT && !FPSEP) {   // the strip buffer is free: the fingerprint's strip goes there
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) load_fp_strips<H, NC>(fp, c0, fpsm, &s_fbar);
  }
  if constexpr (PART != 2) {
    if (act_b) {
      twiddle_tab<RB, RA, false, 1>(v, j);
      DftP<RB, false>::run(v[0]);
    }
  }

  if constexpr (PART == 1) {
    __syncthreads();
    if (act_b) {
      float2* dst = sm + j * NC + c;
#pragma unroll
      for (int r = 0; r < RB; ++r) dst[r * RA * NC] = v[0][r];
    }
  } else {
    // fingerprint bin i of the strip's first column
    auto fp_bin0 = [&](int i) -> float2 {
      const char* p = FPT ? fpsm : static_cast<const char*>(fp.spec);
      if (fp32) return reinterpret_cast<const float2*>(p)[i * 4];
      return __half22float2(reinterpret_cast<const __half2*>(p)[i * 4]);
    };
    if constexpr (FPT) {
      if (!block_wait(&s_fbar, 0, a.err)) return;
    } else {
      __syncthreads();   // every strip value read
    }
    if (c0 == 0) {
      // packed column 0 (DC + i*Nyquist): the product needs bin H - i as
      // well, through two scratch columns (in the strip buffer where it is
      // free): the bins, and each thread's products
      float2* X0 = FPT && !FPSEP ? reinterpret_cast<float2*>(reinterpret_cast<char*>(sm) + col_buf_bytes<CP>(NC)) : sm;
      if (c == 0 && act_b) {
#pragma unroll
        for (int r = 0; r < RB; ++r) X0[j + r * RA] = v[0][r];
      }
      __syncthreads();
      if (c == 0 && act_b) {
#pragma unroll 1
        for (int i = j; i < H; i += RA) {
          const int im = i == 0 ? 0 : H - i;
          X0[H + i] = packed_col0_product(X0[i], X0[im], fp_bin0(i), fp_bin0(im));
        }
#pragma unroll
        for (int r = 0; r < RB; ++r) v[0][r] = X0[H + j + r * RA];
      }
      __syncthreads();
    }
    if (act_b && col != 0) {
      // this thread's bins, in shared memory or the spectrum's own strips
      const int e0 = ((FPT ? c >> 2 : 0) * H + j) * 4 + (c & 3);
      const char* f = FPT ? fpsm + (c >> 2) * fp_strip_pad(NC)
                          : static_cast<const char*>(fp.spec) + (size_t)(col >> 2) * (H * 4 * (fp32 ? 8 : 4));
      if (fp32) {
        const float2* p = reinterpret_cast<const float2*>(f) + e0;
#pragma unroll
        for (int r = 0; r < RB; ++r) v[0][r] = c_conj_mul(v[0][r], FPT ? p[r * RA * 4] : __ldg(p + r * RA * 4));
      } else {
        const __half2* p = reinterpret_cast<const __half2*>(f) + e0;
#pragma unroll
        for (int r = 0; r < RB; ++r)
          v[0][r] = c_conj_mul(v[0][r], __half22float2(FPT ? p[r * RA * 4] : __ldg(p + r * RA * 4)));
      }
    }
    if (FPT && !FPSEP) __syncthreads();   // every fingerprint bin read before the buffer is rewritten
    if (act_b) {
      DftP<RB, true>::run(v[0]);
      float2* dst = sm + j * LB * NC + c;
#pragma unroll
      for (int r = 0; r < RB; ++r) dst[r * NC] = v[0][r];
    }
    __syncthreads();
    float2 u[1][RA];
    if (act_a) {
      const float2* src = sm + j * NC + c;
#pragma unroll
      for (int r = 0; r < RA; ++r) u[0][r] = src[r * LB * NC];
    }
    if constexpr (TMA) __syncthreads();
    if (act_a) {
      twiddle_tab<RA, RB, true, 1>(u, j);
      DftP<RA, true>::run(u[0]);
      float2* dst = TMA ? sm + j * NC + c : Z + (size_t)j * Wh + col;
#pragma unroll
      for (int r = 0; r < RA; ++r) dst[(size_t)r * RB * (TMA ? NC : Wh)] = u[0][r];
    }
  }
  if constexpr (TMA) {
    fence_proxy_async_smem();
    __syncthreads();
    if (t == 0) {
#pragma unroll 1
      for (int b = 0; b < H / BR; ++b) tma_store_2d(map, 2 * c0, ws * H + b * BR, sm + b * BR * NC);
      bulk_commit();
      bulk_wait_read();
    }
  }
}

}  // namespace

}  // namespace prnu
