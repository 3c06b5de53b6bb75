// residual.cu -- noise residual of uint8 frames (Sec. 2.2, W(I) = I - F(I)),
// F = 3x3 local Wiener filter with the frame's mean local variance as the
// noise power, borders replicated.
//
// The 3x3 moments of uint8 pixels are integers: S1 = sum x, S2 = sum x^2,
// V = 9 S2 - S1^2 = 81 * (population variance), D = 9 x - S1 = 9 (x - mu).
// The frame noise power nu2 = sum V / (81 H W) is accumulated exactly in
// 64-bit integers, so it does not depend on the reduction order.  Then
//   W = (x - mu) nu2 / var = 9 D nu2 / V   where var >= nu2 (and V > 0),
//   W = x - mu = D / 9                      elsewhere,
// and R = x W (PRNU_WEIGHT_BY_INTENSITY) or W.
#include <algorithm>
#include <type_traits>

#include "internal.h"

namespace prnu {

namespace {

// A thread covers 4 adjacent pixels of RPT rows, a block of 32 x 8 threads a
// tile of 128 x 8*RPT.  Everything up to V and D is an integer below 2^24, so
// it is computed exactly in FP32, two pixels to a packed instruction, the 3x3
// sums as sums over rows (kept for the next row), then over columns.  Against
// one pixel per thread from a shared-memory tile with 9 integer loads a pixel,
// 30 full-HD frames to normalised FP16 (three passes, the frames in L2) take
// 246 us instead of 737; what bounds it is instruction issue (63%),
// 34 instructions a pixel and pass.
constexpr int kBX = 32, kPX = 4;   // lanes of a block's row, pixels of a thread
constexpr int kMomentFrames = 1024;   // frames of the estimate whose noise powers one launch sums

// rows per thread: 8, but 2 where 8 would leave the GPU's 152 SMs with less
// than two blocks each
inline int resid_rows(int F, int H, int W) {
  const long long blocks = (long long)F * ((W + kBX * kPX - 1) / (kBX * kPX)) * ((H + 63) / 64);
  return blocks >= 304 ? 8 : 2;
}
inline dim3 resid_grid(int F, int H, int W, int rpt) {
  return dim3((W + kBX * kPX - 1) / (kBX * kPX), (H + 8 * rpt - 1) / (8 * rpt), F);
}

// byte i of w as a float: the byte in the low mantissa bits of 2^23, minus 2^23
template <int I>
__device__ __forceinline__ float byte_f(uint32_t w) {
  return __uint_as_float(__byte_perm(w, 0x4B000000u, 0x7440 | I));
}

// Pixels x-1 .. x+4 of one row (borders replicated): the middle four as two
// packed pairs, the outer two apart.
struct Row6 {
  float2 a, b;   // (x, x+1), (x+2, x+3)
  float l, r;    // x-1, x+4
};
struct Raw6 {    // the same as bytes: x .. x+3, x-1, x+4
  uint32_t w, l, r;
};
// VEC: rows are 4-byte aligned (x is a multiple of 4)
template <bool VEC>
__device__ __forceinline__ Raw6 load_raw6(const uint8_t* __restrict__ row, int x, int W) {
  Raw6 o;
  if (VEC && x + 3 < W) {
    o.w = __ldg(reinterpret_cast<const uint32_t*>(row + x));
  } else {
    o.w = __ldg(row + min(x, W - 1)) | (uint32_t)__ldg(row + min(x + 1, W - 1)) << 8 |
          (uint32_t)__ldg(row + min(x + 2, W - 1)) << 16 | (uint32_t)__ldg(row + min(x + 3, W - 1)) << 24;
  }
  o.l = __ldg(row + min(max(x - 1, 0), W - 1));
  o.r = __ldg(row + min(x + 4, W - 1));
  return o;
}
__device__ __forceinline__ Row6 row_floats(const Raw6& q) {
  const float2 m = make_float2(-8388608.f, -8388608.f);
  Row6 o;
  o.a = __fadd2_rn(make_float2(byte_f<0>(q.w), byte_f<1>(q.w)), m);
  o.b = __fadd2_rn(make_float2(byte_f<2>(q.w), byte_f<3>(q.w)), m);
  o.l = byte_f<0>(q.l) - 8388608.f;
  o.r = byte_f<0>(q.r) - 8388608.f;
  return o;
}
__device__ __forceinline__ Row6 row_square(const Row6& p) {
  return Row6{__fmul2_rn(p.a, p.a), __fmul2_rn(p.b, p.b), p.l * p.l, p.r * p.r};
}
__device__ __forceinline__ Row6 row_add(const Row6& p, const Row6& q) {
  return Row6{__fadd2_rn(p.a, q.a), __fadd2_rn(p.b, q.b), p.l + q.l, p.r + q.r};
}
// sums of three adjacent columns around each of the four pixels
__device__ __forceinline__ void row_sum3(const Row6& c, float2& a, float2& b) {
  const float u = c.a.x + c.a.y, v = c.b.x + c.b.y;
  a = make_float2(c.l + u, u + c.b.x);
  b = make_float2(c.a.y + v, v + c.r);
}

// V (and with D the centre's offset) of the four pixels of RPT rows, row by row
// to fn(k, the row's pixels, Va, Vb, Da, Db); row(i) gives row i - 1 (0 <= i <
// RPT + 2).
template <int RPT, class Rows, class Fn>
__device__ __forceinline__ void for_rows(Rows&& row, Fn&& fn) {
  const Row6 up = row(0);
  Row6 mid = row(1);
  Row6 s1 = row_add(up, mid), s2 = row_add(row_square(up), row_square(mid));   // of the two rows above the next
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    const Row6 dn = row(k + 2), dn2 = row_square(dn);
    float2 a1, b1, a2, b2;
    row_sum3(row_add(s1, dn), a1, b1);
    row_sum3(row_add(s2, dn2), a2, b2);
    const float2 nine = make_float2(9.f, 9.f);
    const float2 na1 = make_float2(-a1.x, -a1.y), nb1 = make_float2(-b1.x, -b1.y);
    fn(k, mid, __ffma2_rn(nine, a2, __fmul2_rn(na1, a1)), __ffma2_rn(nine, b2, __fmul2_rn(nb1, b1)),
       __ffma2_rn(nine, mid.a, na1), __ffma2_rn(nine, mid.b, nb1));
    s1 = row_add(mid, dn);
    s2 = row_add(row_square(mid), dn2);
    mid = dn;
  }
}

// rows y0 - 1 .. of the frame f, its first and last rows repeated outside
template <bool VEC>
struct FrameRows {
  const uint8_t* f;
  size_t pitch;
  int H, W, x, y0;
  __device__ __forceinline__ Raw6 raw(int i) const {
    return load_raw6<VEC>(f + (size_t)min(max(y0 - 1 + i, 0), H - 1) * pitch, x, W);
  }
  __device__ __forceinline__ Row6 operator()(int i) const { return row_floats(raw(i)); }
};

// per block: the integer sum of 81 * (local variance) of its pixels, one slot per block
template <int RPT, bool VEC>
__global__ void __launch_bounds__(kBX * 8) k_resid_moments(const uint8_t* __restrict__ frames, size_t pitch, int H,
                                                           int W, unsigned long long* __restrict__ part_out) {
  __shared__ unsigned long long part[8];
  const int f = blockIdx.z, tx = threadIdx.x;
  const int x = (blockIdx.x * kBX + tx) * kPX, y0 = (blockIdx.y * 8 + threadIdx.y) * RPT;
  unsigned acc = 0;   // at most 32 terms of at most 81 * 255^2 / 4 each
  if (x < W && y0 < H) {
    for_rows<RPT>(FrameRows<VEC>{frames + (size_t)f * H * pitch, pitch, H, W, x, y0},
                       [&](int k, const Row6&, float2 va, float2 vb, float2, float2) {
                         if (y0 + k >= H) return;
                         if (x + 3 < W) {   // four terms: exact below 2^24
                           acc += __float2uint_rn((va.x + va.y) + (vb.x + vb.y));
                         } else {
                           acc += __float2uint_rn(va.x + (x + 1 < W ? va.y : 0.f) + (x + 2 < W ? vb.x : 0.f));
                         }
                       });
  }
  unsigned long long v = acc;
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (tx == 0) part[threadIdx.y] = v;
  __syncthreads();
  if (threadIdx.y == 0 && tx == 0) {
    unsigned long long s = 0;
    for (int k = 0; k < 8; ++k) s += part[k];
    part_out[(size_t)f * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x] = s;
  }
}

// one block per frame: acc[f] = sum of the frame's block slots (integers: exact in any order)
__global__ void k_resid_noise(const unsigned long long* __restrict__ part, int nblk,
                              unsigned long long* __restrict__ acc) {
  __shared__ unsigned long long red[32];
  const int f = blockIdx.x;
  unsigned long long v = 0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) v += part[(size_t)f * nblk + k];
#pragma unroll
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long t = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += red[k];
    acc[f] = t;
  }
}

// W of one pixel: 9 D nu2 / V or D / 9 (see the head of this file), correctly
// rounded as V <= 20 * 255^2
__device__ __forceinline__ float residual_w(float V, float D, float nu2, float nu2x81) {
  const bool wiener = V > 0.f && V >= nu2x81;
  return refined_quotient(wiener ? (9.f * D) * nu2 : D, wiener ? V : 9.f);
}

// the frame's noise power and 81 times it, from its integer sum
__device__ __forceinline__ float2 noise_power(unsigned long long acc, int H, int W) {
  const double nu2d = (double)acc / (81.0 * (double)H * (double)W);
  return make_float2((float)nu2d, (float)(81.0 * nu2d));
}

template <int DT>
__device__ __forceinline__ void store4(void* p, size_t o, float4 v, int n, bool vec) {
  if (vec && n >= 4) {
    if constexpr (DT == kF32) {
      *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + o) = v;
    } else {
      uint2 u;
      if constexpr (DT == kF16) {
        const __half2 a = __floats2half2_rn(v.x, v.y), b = __floats2half2_rn(v.z, v.w);
        u = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      } else {
        const __nv_bfloat162 a = __floats2bfloat162_rn(v.x, v.y), b = __floats2bfloat162_rn(v.z, v.w);
        u = make_uint2(*reinterpret_cast<const uint32_t*>(&a), *reinterpret_cast<const uint32_t*>(&b));
      }
      *reinterpret_cast<uint2*>(reinterpret_cast<uint16_t*>(p) + o) = u;
    }
  } else {
    store_store_type<DT>(p, o, v.x);
    if (n > 1) store_store_type<DT>(p, o + 1, v.y);
    if (n > 2) store_store_type<DT>(p, o + 2, v.z);
    if (n > 3) store_store_type<DT>(p, o + 3, v.w);
  }
}

// MODE 0: store R (and scale[f] = 1); MODE 1: per-block sum of R^2 (double) to
// partials; MODE 2: store R * scale[f].
// R(y, x) of frame f goes to out[f * lay.fpitch + lay.roff + y * lay.rpitch + x];
// vec_out: the quads of a row lie on vector boundaries.
template <int DT, int MODE, int RPT, bool VEC>
__global__ void __launch_bounds__(kBX * 8) k_resid_apply(const uint8_t* __restrict__ frames, size_t pitch, int H,
                                                         int W, const unsigned long long* __restrict__ acc,
                                                         int weight, void* __restrict__ out,
                                                         double* __restrict__ partials, float* __restrict__ scale,
                                                         ResidLayout lay, bool vec_out) {
  constexpr int NS = RPT < 4 ? RPT : 4;
  __shared__ double part[MODE == 1 ? 8 * NS : 1];
  __shared__ float2 s_nu2;
  const int f = blockIdx.z, tx = threadIdx.x;
  if (tx == 0 && threadIdx.y == 0) s_nu2 = noise_power(acc[f], H, W);   // once per block: the FP64 pipe is narrow
  __syncthreads();
  const float2 nu2 = s_nu2;
  const float s = MODE == 2 ? scale[f] : 1.f;
  const int x = (blockIdx.x * kBX + tx) * kPX, y0 = (blockIdx.y * 8 + threadIdx.y) * RPT;
  float sq[NS];   // of rows k, k + NS
#pragma unroll
  for (int k = 0; k < NS; ++k) sq[k] = 0.f;
  if (x < W && y0 < H) {
    for_rows<RPT>(FrameRows<VEC>{frames + (size_t)f * H * pitch, pitch, H, W, x, y0},
                       [&](int k, const Row6& p, float2 va, float2 vb, float2 da, float2 db) {
                         if (y0 + k >= H) return;
                         float4 r = make_float4(residual_w(va.x, da.x, nu2.x, nu2.y), residual_w(va.y, da.y, nu2.x, nu2.y),
                                                residual_w(vb.x, db.x, nu2.x, nu2.y), residual_w(vb.y, db.y, nu2.x, nu2.y));
                         if (weight) r = make_float4(p.a.x * r.x, p.a.y * r.y, p.b.x * r.z, p.b.y * r.w);
                         if (MODE == 1) {
                           if (x + 1 >= W) r.y = 0.f;
                           if (x + 2 >= W) r.z = 0.f;
                           if (x + 3 >= W) r.w = 0.f;
                           sq[k % NS] += fmaf(r.x, r.x, r.y * r.y) + fmaf(r.z, r.z, r.w * r.w);
                         } else {
                           if (MODE == 2) r = make_float4(r.x * s, r.y * s, r.z * s, r.w * s);
                           store4<DT>(out, (size_t)f * lay.fpitch + lay.roff + (size_t)(y0 + k) * lay.rpitch + x, r, W - x,
                                      vec_out);
                         }
                       });
  }
  if (MODE == 0 && scale && blockIdx.x == 0 && blockIdx.y == 0 && tx == 0 && threadIdx.y == 0) scale[f] = 1.f;
  if constexpr (MODE == 1) {   // float over a warp's 128 pixels of one or two rows, double beyond
    const double t = block_sum(sq, tx, threadIdx.y, part);
    if (threadIdx.y == 0 && tx == 0)
      partials[(size_t)f * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

// one block per frame: fixed-order sum of the block partials, s = 1/RMS
__global__ void k_resid_scale(const double* __restrict__ partials, int nblk, int H, int W, float* __restrict__ scale) {
  __shared__ double part[32];
  const int f = blockIdx.x;
  double s = 0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) s += partials[(size_t)f * nblk + k];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += part[k];
    const double ms = t / ((double)H * (double)W);
    scale[f] = ms > 0 ? (float)(1.0 / sqrt(ms)) : 1.f;
  }
}

__global__ void k_fill(float* __restrict__ p, int n, float v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) p[i] = v;
}

// Copy of dense [F][H][W] frames into the zero-bordered layout: padded row
// yp, column xp of frame f holds pixel (yp - 1, xp - 1), or 0 outside.
template <typename T>
__global__ void k_pad_frames(const T* __restrict__ in, int H, int W, T* __restrict__ out) {
  const int P = W + 3;
  const int xp = blockIdx.x * blockDim.x + threadIdx.x, yp = blockIdx.y;
  const int f = blockIdx.z;
  if (xp >= P) return;
  const int x = xp - 1, y = yp - 1;
  T v{};
  if ((unsigned)x < (unsigned)W && (unsigned)y < (unsigned)H) v = in[((size_t)f * H + y) * W + x];
  out[(size_t)f * (H + 3) * P + (size_t)yp * P + xp] = v;
}

// The same layout for half storage as pairs: element (yp, xp) holds the
// 16-bit values of padded pixels (yp, xp) and (yp, xp + 1) (0 beyond the
// padded row), the first in the low half (the .x of a __half2).
__global__ void k_pad_pairs(const uint16_t* __restrict__ in, int H, int W, uint32_t* __restrict__ out) {
  const int P = W + 3;
  const int xp = blockIdx.x * blockDim.x + threadIdx.x, yp = blockIdx.y;
  const int f = blockIdx.z;
  if (xp >= P) return;
  const int x = xp - 1, y = yp - 1;
  uint32_t lo = 0, hi = 0;
  if ((unsigned)y < (unsigned)H) {
    const uint16_t* row = in + ((size_t)f * H + y) * W;
    if ((unsigned)x < (unsigned)W) lo = row[x];
    if ((unsigned)(x + 1) < (unsigned)W) hi = row[x + 1];
  }
  out[(size_t)f * (H + 3) * P + (size_t)yp * P + xp] = lo | (hi << 16);
}

// the kernel template with its rows per thread and row alignment chosen
template <class Fn>
void resid_dispatch(int rpt, bool vec, Fn&& fn) {
  using std::integral_constant;
  if (rpt == 8 && vec) fn(integral_constant<int, 8>{}, integral_constant<bool, true>{});
  else if (rpt == 8) fn(integral_constant<int, 8>{}, integral_constant<bool, false>{});
  else if (vec) fn(integral_constant<int, 2>{}, integral_constant<bool, true>{});
  else fn(integral_constant<int, 2>{}, integral_constant<bool, false>{});
}
bool rows_aligned4(const void* frames, size_t pitch) { return ((reinterpret_cast<uintptr_t>(frames) | pitch) & 3) == 0; }

template <int MODE>
void apply_dispatch(int dtype, int rpt, bool vec, dim3 g, cudaStream_t s, const uint8_t* frames, size_t pitch, int H,
                    int W, const unsigned long long* acc, int weight, void* out, double* partials, float* scale,
                    const ResidLayout& l) {
  const dim3 b(kBX, 8);
  // quads start at multiples of 4 elements of rows and frames that do too
  const bool vec_out = out && (l.roff | l.rpitch | l.fpitch) % 4 == 0 &&
                       reinterpret_cast<uintptr_t>(out) % (dtype == kF32 ? 16 : 8) == 0;
  resid_dispatch(rpt, vec, [&](auto R, auto V) {
    constexpr int RPT = decltype(R)::value;
    constexpr bool VEC = decltype(V)::value;
    auto* fn = k_resid_apply<kF32, MODE, RPT, VEC>;
    if constexpr (MODE != 1) {   // MODE 1 stores no residual
      if (dtype == kF16) fn = k_resid_apply<kF16, MODE, RPT, VEC>;
      else if (dtype == kBF16) fn = k_resid_apply<kBF16, MODE, RPT, VEC>;
    }
    fn<<<g, b, 0, s>>>(frames, pitch, H, W, acc, weight, out, partials, scale, l, vec_out);
  });
  PRNU_CUDA_TRY(cudaGetLastError());
}

// the frames' integer variance sums, block slots first
void launch_moments(const uint8_t* frames, int F, int H, int W, size_t pitch, int rpt, unsigned long long* slots,
                    unsigned long long* acc, cudaStream_t s, LaunchCounter& lc) {
  const dim3 g = resid_grid(F, H, W, rpt);
  resid_dispatch(rpt, rows_aligned4(frames, pitch), [&](auto R, auto V) {
    k_resid_moments<decltype(R)::value, decltype(V)::value><<<g, dim3(kBX, 8), 0, s>>>(frames, pitch, H, W, slots);
  });
  PRNU_CUDA_TRY(cudaGetLastError());
  k_resid_noise<<<F, 256, 0, s>>>(slots, (int)(g.x * g.y), acc);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n += 2;
}

// K = sum_l I W(I) / sum_l I^2 (Eq. 2) of a thread's pixels over all L frames.
// The numerator is a compensated FP32 sum (48 bits; the FP64 pipe takes 1/64 of
// the FP32 rate), the denominator an integer: exact in FP32 over up to 256
// frames, which LONG then adds to a compensated sum.  Against 64 bits K is off
// by 3.9e-8, 2.8e-8 and 2.5e-8 of its 2-norm for 1, 16 and 1000 frames (with
// rounded products and FP64 sums 4.5e-8, 2.9e-8, 2.5e-8).  One pass over the frames
// where residuals in memory and FP64 sums took three and two more: 0.58 ms (with the noise powers)
// instead of 2.98 for 16 frames of 4000 x 3000, bound by issue (59%).
template <bool VEC, bool LONG>
__global__ void __launch_bounds__(kBX * 8, 2) k_fp_estimate(const uint8_t* __restrict__ frames, size_t pitch, int L,
                                                         int H, int W, const unsigned long long* __restrict__ acc,
                                                         float* __restrict__ K, bool vec_out) {
  constexpr int RPT = 2;
  __shared__ float2 s_nu2[256];
  const int tx = threadIdx.x, tid = threadIdx.y * kBX + tx;
  const int x = (blockIdx.x * kBX + tx) * kPX, y0 = (blockIdx.y * 8 + threadIdx.y) * RPT;
  const float2 zero = make_float2(0.f, 0.f);
  float2 n[RPT][2], nc[RPT][2], d[RPT][2], dh[RPT][2], dl[RPT][2];
#pragma unroll
  for (int k = 0; k < RPT; ++k)
#pragma unroll
    for (int q = 0; q < 2; ++q) n[k][q] = nc[k][q] = dh[k][q] = dl[k][q] = zero;
  for (int l0 = 0; l0 < L; l0 += 256) {
    const int lc = min(256, L - l0);
    __syncthreads();
    if (tid < lc) s_nu2[tid] = noise_power(acc[l0 + tid], H, W);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < RPT; ++k) d[k][0] = d[k][1] = zero;
    if (x < W && y0 < H) {
      FrameRows<VEC> rows{frames + (size_t)l0 * H * pitch, pitch, H, W, x, y0};
      Raw6 next[RPT + 2];   // the next frame's rows are loaded before this one's are used
#pragma unroll
      for (int i = 0; i < RPT + 2; ++i) next[i] = rows.raw(i);
      for (int l = 0; l < lc; ++l) {
        const float2 nu2 = s_nu2[l];
        Raw6 cur[RPT + 2];
#pragma unroll
        for (int i = 0; i < RPT + 2; ++i) cur[i] = next[i];
        if (l + 1 < lc) {
          rows.f += (size_t)H * pitch;
#pragma unroll
          for (int i = 0; i < RPT + 2; ++i) next[i] = rows.raw(i);
        }
        for_rows<RPT>([&](int i) { return row_floats(cur[i]); },
                           [&](int k, const Row6& p, float2 va, float2 vb, float2 da, float2 db) {
                             const float2 wa = make_float2(residual_w(va.x, da.x, nu2.x, nu2.y),
                                                           residual_w(va.y, da.y, nu2.x, nu2.y));
                             const float2 wb = make_float2(residual_w(vb.x, db.x, nu2.x, nu2.y),
                                                           residual_w(vb.y, db.y, nu2.x, nu2.y));
                             csum_add2(n[k][0], nc[k][0], __fmul2_rn(p.a, wa));
                             csum_add2(n[k][1], nc[k][1], __fmul2_rn(p.b, wb));
                             d[k][0] = __ffma2_rn(p.a, p.a, d[k][0]);
                             d[k][1] = __ffma2_rn(p.b, p.b, d[k][1]);
                           });
      }
    }
#pragma unroll
    for (int k = 0; k < RPT; ++k)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (LONG) csum_add2(dh[k][q], dl[k][q], d[k][q]);
        else dh[k][q] = d[k][q];
      }
  }
  if (x >= W) return;
  // (s + c) / (h + l): a quotient and one correction by its remainder
  auto ratio = [](float s, float c, float h, float l) {
    if (!(h > 0.f)) return 0.f;
    const float q = s / h;
    return q + (fmaf(-q, h, s) + fmaf(-q, l, c)) / h;
  };
#pragma unroll
  for (int k = 0; k < RPT; ++k) {
    if (y0 + k >= H) break;
    const float4 r = make_float4(ratio(n[k][0].x, nc[k][0].x, dh[k][0].x, dl[k][0].x),
                                 ratio(n[k][0].y, nc[k][0].y, dh[k][0].y, dl[k][0].y),
                                 ratio(n[k][1].x, nc[k][1].x, dh[k][1].x, dl[k][1].x),
                                 ratio(n[k][1].y, nc[k][1].y, dh[k][1].y, dl[k][1].y));
    store4<kF32>(K, (size_t)(y0 + k) * W + x, r, W - x, vec_out);
  }
}

// ---------------------------------------------------------------- frame-literal residuals (Sec. 3.2)
//
// The paper warps the frame for every candidate and extracts the residual of
// the warped frame.  For render r (source frame f, similarity a11..a22):
//   X(p)  = bilinear(I_f, c + A (p - c)), each tap outside the frame 0,
//   W(X)  = X - Wiener3x3(X), 3x3 moments with replicated borders, noise power
//           nu2 = mean over the frame of the local variances of X,
//   R     = X W(X) (PRNU_WEIGHT_BY_INTENSITY) or W(X).
// X is not an integer image, so the moments are taken in float from the
// differences to the window's centre (d = x_k - x_c: mean m1 = sum d / 9,
// variance sum d^2 / 9 - m1^2), which keeps the cancellation small.  A block
// warps a 64 x 64 tile plus a one-pixel halo into shared memory; halo pixels
// outside the frame are the warped values at the clamped position (the
// replicated border).  A thread takes two adjacent columns, packed, down 8
// rows.  At 1080p a render takes 6.3 us of warp and moments and 3.3 us
// of residual (one pixel a thread from shared memory and general bounds tests
// everywhere: 11.4 and 7.4), both bound by issue.

constexpr int kLX = 64, kLY = 64, kLR = 8;
constexpr int kLP = kLX + 4, kLTY = kLY + 2;   // tile pitch and rows: pixel (x, y) of the tile at (x + 2, y + 1)
static_assert(kLX == 2 * 32 && kLY == 8 * kLR, "a lane takes a column pair, each of 8 warps kLR rows");

// uint8 -> float without a conversion instruction: the byte in the low
// mantissa bits of 2^23 (exact for every byte value)
__device__ __forceinline__ float u8f(uint32_t v) { return __int_as_float(0x4B000000u | v) - 8388608.f; }

__device__ __forceinline__ float warp_u8(const uint8_t* __restrict__ fr, int pitch, int H, int W, const WorkItem& it,
                                         float cx, float cy, int x, int y) {
  const float dx = (float)x - cx, dy = (float)y - cy;
  const float qx = fmaf(it.a11, dx, fmaf(it.a12, dy, cx));
  const float qy = fmaf(it.a21, dx, fmaf(it.a22, dy, cy));
  const float fx0 = floorf(qx), fy0 = floorf(qy);
  // every tap outside (also keeps the int conversion in range)
  if (!(fx0 >= -1.f && fx0 <= (float)(W - 1) && fy0 >= -1.f && fy0 <= (float)(H - 1))) return 0.f;
  const float fx = qx - fx0, fy = qy - fy0;
  const int x0 = (int)fx0, y0 = (int)fy0;
  const bool xa = x0 >= 0, xb = x0 + 1 < W, ya = y0 >= 0, yb = y0 + 1 < H;
  const uint8_t* r0 = fr + (ya ? y0 : 0) * pitch;
  const uint8_t* r1 = fr + (yb ? y0 + 1 : 0) * pitch;
  const float v00 = (ya && xa) ? u8f(__ldg(r0 + x0)) : 0.f;
  const float v01 = (ya && xb) ? u8f(__ldg(r0 + x0 + 1)) : 0.f;
  const float v10 = (yb && xa) ? u8f(__ldg(r1 + x0)) : 0.f;
  const float v11 = (yb && xb) ? u8f(__ldg(r1 + x0 + 1)) : 0.f;
  const float top = fmaf(fx, v01, (1.f - fx) * v00), bot = fmaf(fx, v11, (1.f - fx) * v10);
  return fmaf(fy, bot, (1.f - fy) * top);
}

// warp_u8 where the four taps lie inside the frame: floor(q) by rounding q - 1/2
// to an integer at 1.5 * 2^23 (an integer q may give q - 1 and weight 1 on its
// own tap: the same value), whose mantissa holds the tap's index
__device__ __forceinline__ float warp_u8_inside(const uint8_t* __restrict__ fr, int pitch, float qx, float qy) {
  constexpr float kRound = 12582912.f;
  constexpr int kBits = 0x4B400000;
  const float tx = (qx - 0.5f) + kRound, ty = (qy - 0.5f) + kRound;
  const float fx = qx - (tx - kRound), fy = qy - (ty - kRound);
  const uint8_t* p = fr + ((__float_as_int(ty) - kBits) * pitch + (__float_as_int(tx) - kBits));
  const uint8_t* r = p + pitch;
  const float v00 = u8f(__ldg(p)), v01 = u8f(__ldg(p + 1)), v10 = u8f(__ldg(r)), v11 = u8f(__ldg(r + 1));
  const float top = fmaf(fx, v01 - v00, v00), bot = fmaf(fx, v11 - v10, v10);
  return fmaf(fy, bot - top, top);
}

// Window mean offset m1 and population variance of a column pair's pixels,
// from the rows above, at and below: l, c, r the pairs (x-1, x), (x, x+1) and
// (x+1, x+2).
struct PairRow {
  float2 l, c, r;
};
__device__ __forceinline__ void pair_moments(const PairRow& up, const PairRow& mid, const PairRow& dn, float2& m1,
                                             float2& var) {
  const float2 nc = make_float2(-mid.c.x, -mid.c.y);
  float2 s1 = make_float2(0.f, 0.f), s2 = s1;
  auto term = [&](float2 v) {
    const float2 d = __fadd2_rn(v, nc);
    s1 = __fadd2_rn(s1, d);
    s2 = __ffma2_rn(d, d, s2);
  };
  term(up.l);
  term(up.c);
  term(up.r);
  term(mid.l);
  term(mid.r);
  term(dn.l);
  term(dn.c);
  term(dn.r);
  const float2 ninth = make_float2(1.f / 9.f, 1.f / 9.f);
  m1 = __fmul2_rn(s1, ninth);
  var = __ffma2_rn(make_float2(-m1.x, -m1.y), m1, __fmul2_rn(s2, ninth));
}

// per block: sum of the local variances of its pixels (double), one slot per
// block; the warped frame itself to X[r][H][W] for the second pass
__global__ void __launch_bounds__(256) k_lit_moments(const uint8_t* __restrict__ frames, size_t pitch, int H, int W,
                                                     const WorkItem* __restrict__ renders,
                                                     double* __restrict__ partials, float* __restrict__ X) {
  __shared__ __align__(16) float tile[kLTY * kLP];
  __shared__ double part[8 * 4];
  const WorkItem it = renders[blockIdx.z];
  const uint8_t* fr = frames + (size_t)it.frame * H * pitch;
  const float cx = 0.5f * (float)(W - 1), cy = 0.5f * (float)(H - 1);
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int x0 = blockIdx.x * kLX, y0 = blockIdx.y * kLY;
  const int xa = max(x0 - 1, 0), xb = min(x0 + kLX, W - 1), ya = max(y0 - 1, 0), yb = min(y0 + kLY, H - 1);
  auto map = [&](int x, int y, float& qx, float& qy) {
    const float dx = (float)x - cx, dy = (float)y - cy;
    qx = fmaf(it.a11, dx, fmaf(it.a12, dy, cx));
    qy = fmaf(it.a21, dx, fmaf(it.a22, dy, cy));
  };
  // the map is affine: its corners bound the tile
  bool inside = true;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    float qx, qy;
    map(k & 1 ? xb : xa, k & 2 ? yb : ya, qx, qy);
    inside = inside && qx >= 1.5f && qx <= (float)W - 2.5f && qy >= 1.5f && qy <= (float)H - 2.5f;
  }
  auto sample = [&](int sx, int sy) {   // tile pixel (sx - 1, sy - 1)
    const int x = min(max(x0 + sx - 1, 0), W - 1), y = min(max(y0 + sy - 1, 0), H - 1);
    float v;
    if (inside) {
      float qx, qy;
      map(x, y, qx, qy);
      v = warp_u8_inside(fr, (int)pitch, qx, qy);
    } else {
      v = warp_u8(fr, (int)pitch, H, W, it, cx, cy, x, y);
    }
    tile[sy * kLP + sx + 1] = v;
  };
  for (int sy = wp; sy < kLTY; sy += 8) {
    sample(lane + 1, sy);
    sample(lane + 33, sy);
  }
  if (threadIdx.x < 2 * kLTY) sample(threadIdx.x & 1 ? kLX + 1 : 0, threadIdx.x >> 1);   // the two halo columns
  __syncthreads();
  const int x = x0 + 2 * lane, ys = y0 + wp * kLR;
  float2 acc[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
  if (x < W) {   // W is even: both pixels of the pair
    auto row = [&](int k) {   // tile row k of this warp's band (0: the row above it)
      const float2* p = reinterpret_cast<const float2*>(tile + (wp * kLR + k) * kLP) + lane;
      const float2 a = p[0], c = p[1], b = p[2];
      return PairRow{make_float2(a.y, c.x), c, make_float2(c.y, b.x)};
    };
    PairRow up = row(0), mid = row(1);
    float* xo = X + ((size_t)blockIdx.z * H + ys) * W + x;
#pragma unroll
    for (int k = 0; k < kLR; ++k) {
      const PairRow dn = row(k + 2);
      if (ys + k < H) {
        *reinterpret_cast<float2*>(xo + (size_t)k * W) = mid.c;
        float2 m, var;
        pair_moments(up, mid, dn, m, var);
        acc[k & 1] = __fadd2_rn(acc[k & 1], var);
      }
      up = mid;
      mid = dn;
    }
  }
  // float over 128 pixels (4 rows of every other column of the warp's band),
  // double beyond: the FP64 pipe is a small fraction of the FP32 one
  float v[4] = {acc[0].x, acc[0].y, acc[1].x, acc[1].y};
  const double s = block_sum(v, lane, wp, part);
  if (threadIdx.x == 0)
    partials[(size_t)blockIdx.z * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x] = s;
}

// one block per render: nu2 = (fixed-order sum of the block partials) / (H W)
__global__ void k_lit_noise(const double* __restrict__ partials, int nblk, int H, int W, float* __restrict__ nu2) {
  __shared__ double part[32];
  const int r = blockIdx.x;
  double s = 0.0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) s += partials[(size_t)r * nblk + k];
#pragma unroll
  for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) t += part[k];
    nu2[r] = (float)(t / ((double)H * (double)W));
  }
}

// R of every pixel into out[r * lay.fpitch + lay.roff + y * lay.rpitch + x]
// (float) from X, the first pass's warped frame, a column pair and kLR rows to
// a thread, straight from global memory
__global__ void __launch_bounds__(256) k_lit_apply(const float* __restrict__ X, int H, int W,
                                                   const float* __restrict__ nu2, int weight, float* __restrict__ out,
                                                   ResidLayout lay) {
  const int x = blockIdx.x * kLX + 2 * (threadIdx.x & 31), ys = blockIdx.y * kLY + (threadIdx.x >> 5) * kLR;
  if (x >= W || ys >= H) return;
  const float* xr = X + (size_t)blockIdx.z * H * W;
  const int xl = max(x - 1, 0), xh = min(x + 2, W - 1);
  auto row = [&](int y) {
    const float* p = xr + (size_t)min(max(y, 0), H - 1) * W;
    const float2 c = __ldg(reinterpret_cast<const float2*>(p + x));
    return PairRow{make_float2(__ldg(p + xl), c.x), c, make_float2(c.y, __ldg(p + xh))};
  };
  const float n2 = nu2[blockIdx.z];
  auto wiener = [&](float m, float var) {   // x - (mu + (x - mu) gain), x - mu = -m1
    const float den = fmaxf(var, n2);
    const float gain = den > 0.f ? __fdividef(fmaxf(var - n2, 0.f), den) : 1.f;
    return -m * (1.f - gain);
  };
  float* o = out + (size_t)blockIdx.z * lay.fpitch + lay.roff + (size_t)ys * lay.rpitch + x;
  PairRow up = row(ys - 1), mid = row(ys);
#pragma unroll
  for (int k = 0; k < kLR; ++k) {
    if (ys + k >= H) break;
    const PairRow dn = row(ys + k + 1);
    float2 m, var;
    pair_moments(up, mid, dn, m, var);
    float2 w = make_float2(wiener(m.x, var.x), wiener(m.y, var.y));
    if (weight) w = __fmul2_rn(mid.c, w);
    o[0] = w.x;
    o[1] = w.y;
    o += lay.rpitch;
    up = mid;
    mid = dn;
  }
}

// Taps of one axis (Sec. 3's resampling): output sample o at input position
// u = (first + o + 0.5) / scale - 0.5, tent weights max(0, 1 - |j - u| a) with a
// = min(scale, 1), indices clamped to the axis, normalised; a sample's taps of
// nonzero weight first, then zero weights up to T.  In double, one thread per
// sample of both axes (y first).
struct TapAxis {
  int n_in, first, n;
  float* w;
  int* idx;
};
__global__ void k_fp_taps(TapAxis ay, TapAxis ax, double scale, int T) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= ay.n + ax.n) return;
  const bool y = i < ay.n;
  const TapAxis t = y ? ay : ax;
  const int o = y ? i : i - ay.n;
  const double a = fmin(scale, 1.0);
  const double u = ((double)(t.first + o) + 0.5) / scale - 0.5;
  const int lo = (int)floor(u - 1.0 / a);
  double tot = 0.0;
  for (int k = 0; k < T; ++k) tot += fmax(1.0 - fabs((double)(lo + k) - u) * a, 0.0);
  int m = 0;
  for (int k = 0; k < T; ++k) {
    const double v = fmax(1.0 - fabs((double)(lo + k) - u) * a, 0.0);
    if (v == 0.0) continue;
    t.w[(size_t)o * T + m] = (float)(v / tot);
    t.idx[(size_t)o * T + m++] = min(max(lo + k, 0), t.n_in - 1);
  }
  for (; m < T; ++m) t.w[(size_t)o * T + m] = 0.f;
}

// Fingerprint resampling: out(y, x) = sum_a sum_b wy[y][a] wx[x][b] K(iy[y][a], ix[x][b]),
// T taps per axis, the first zero weight ends them (a sample without weight has
// no part in the sum: it may hold an infinity or a NaN).
__global__ void k_fp_resize(const float* __restrict__ K, size_t pitch, const float* __restrict__ wy,
                            const int* __restrict__ iy, const float* __restrict__ wx, const int* __restrict__ ix,
                            int T, int H, int W, float* __restrict__ out) {
  const int x = blockIdx.x * blockDim.x + threadIdx.x, y = blockIdx.y;
  if (x >= W) return;
  float acc = 0.f;
  for (int a = 0; a < T; ++a) {
    const float w = wy[(size_t)y * T + a];
    if (w == 0.f) break;
    const float* row = K + (size_t)iy[(size_t)y * T + a] * pitch;
    float r = 0.f;
    for (int b = 0; b < T; ++b) {
      const float v = wx[(size_t)x * T + b];
      if (v == 0.f) break;
      r = fmaf(v, __ldg(row + ix[(size_t)x * T + b]), r);
    }
    acc = fmaf(w, r, acc);
  }
  out[(size_t)y * W + x] = acc;
}

}  // namespace

void launch_fp_estimate(const uint8_t* frames, size_t pitch, int L, int H, int W, unsigned long long* slots,
                        unsigned long long* acc, float* K, cudaStream_t s, LaunchCounter& lc) {
  ProfScope ps(lc, kKindResidual, s);
  // frames are a grid dimension of at most 65535: the noise powers come in
  // runs of kMomentFrames, which reuse the slots of the first
  const int rpt = resid_rows(std::min(L, kMomentFrames), H, W);
  for (int l0 = 0; l0 < L; l0 += kMomentFrames)
    launch_moments(frames + (size_t)l0 * H * pitch, std::min(kMomentFrames, L - l0), H, W, pitch, rpt, slots, acc + l0, s,
                   lc);
  const dim3 g = resid_grid(1, H, W, 2), b(kBX, 8);
  const bool vec = rows_aligned4(frames, pitch), lng = L > 256;
  const bool vec_out = W % 4 == 0 && reinterpret_cast<uintptr_t>(K) % 16 == 0;
  auto* fn = lng ? (vec ? k_fp_estimate<true, true> : k_fp_estimate<false, true>)
                 : (vec ? k_fp_estimate<true, false> : k_fp_estimate<false, false>);
  fn<<<g, b, 0, s>>>(frames, pitch, L, H, W, acc, K, vec_out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}

void launch_pad_frames(const void* in, int dtype, int F, int H, int W, void* out, cudaStream_t s, LaunchCounter& lc,
                       int layout) {
  if (F == 0) return;
  ProfScope ps(lc, kKindResidual, s);
  const dim3 b(256), g((W + 3 + 255) / 256, H + 3, F);
  if (layout == 1 && dtype != kF32)
    k_pad_pairs<<<g, b, 0, s>>>(reinterpret_cast<const uint16_t*>(in), H, W, reinterpret_cast<uint32_t*>(out));
  else if (dtype == kF32)
    k_pad_frames<float><<<g, b, 0, s>>>(reinterpret_cast<const float*>(in), H, W, reinterpret_cast<float*>(out));
  else
    k_pad_frames<uint16_t><<<g, b, 0, s>>>(reinterpret_cast<const uint16_t*>(in), H, W,
                                           reinterpret_cast<uint16_t*>(out));
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}


void launch_literal_residuals(const uint8_t* frames, size_t pitch, int H, int W, const WorkItem* renders, int nr,
                              int weight, float* out, const ResidLayout& lay, float* X, double* partials,
                              float* nu2, cudaStream_t s, LaunchCounter& lc) {
  if (nr == 0) return;
  ProfScope ps(lc, kKindResidual, s);
  const dim3 b(256), g((W + kLX - 1) / kLX, (H + kLY - 1) / kLY, nr);
  k_lit_moments<<<g, b, 0, s>>>(frames, pitch, H, W, renders, partials, X);
  PRNU_CUDA_TRY(cudaGetLastError());
  k_lit_noise<<<nr, 256, 0, s>>>(partials, (int)(g.x * g.y), H, W, nu2);
  PRNU_CUDA_TRY(cudaGetLastError());
  k_lit_apply<<<g, b, 0, s>>>(X, H, W, nu2, weight, out, lay);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n += 3;
}

size_t literal_partials_needed(int nr, int H, int W) {
  return (size_t)nr * ((W + kLX - 1) / kLX) * ((H + kLY - 1) / kLY);
}

size_t fp_estimate_slots(int L, int H, int W) { return residual_partials_needed(std::min(L, kMomentFrames), H, W); }

size_t residual_partials_needed(int F, int H, int W) {
  const dim3 g = resid_grid(F, H, W, resid_rows(F, H, W));
  return (size_t)F * g.x * g.y;
}

void launch_residual(const uint8_t* frames, int F, int H, int W, size_t pitch, int flags, int dtype, void* out,
                     float* scale, unsigned long long* acc, double* partials, cudaStream_t s,
                     LaunchCounter& lc, const ResidLayout* lay) {
  const ResidLayout l = lay ? *lay : ResidLayout{W, (size_t)H * W, 0};
  const int rpt = resid_rows(F, H, W);
  const bool vec = rows_aligned4(frames, pitch);
  const dim3 g = resid_grid(F, H, W, rpt);
  const int weight = (flags & PRNU_WEIGHT_BY_INTENSITY) ? 1 : 0;
  ProfScope ps(lc, kKindResidual, s);
  // the block slots go to `partials` (8-byte slots, reused below by PRNU_NORMALISE)
  launch_moments(frames, F, H, W, pitch, rpt, reinterpret_cast<unsigned long long*>(partials), acc, s, lc);
  if (flags & PRNU_NORMALISE) {
    // the sum of squares does not depend on the storage type
    apply_dispatch<1>(kF32, rpt, vec, g, s, frames, pitch, H, W, acc, weight, nullptr, partials, scale, l);
    k_resid_scale<<<F, 256, 0, s>>>(partials, (int)(g.x * g.y), H, W, scale);
    PRNU_CUDA_TRY(cudaGetLastError());
    apply_dispatch<2>(dtype, rpt, vec, g, s, frames, pitch, H, W, acc, weight, out, partials, scale, l);
    lc.n += 3;
  } else {
    apply_dispatch<0>(dtype, rpt, vec, g, s, frames, pitch, H, W, acc, weight, out, partials, scale, l);
    lc.n++;
  }
}

}  // namespace prnu

namespace prnu {
void launch_fp_resize(const float* K, int Hin, int Win, size_t pitch, double scale, int y0, int x0, int T, float* w,
                      int* idx, int H, int W, float* out, cudaStream_t s, LaunchCounter& lc) {
  ProfScope ps(lc, kKindResidual, s);
  const size_t ny = (size_t)H * T;
  k_fp_taps<<<(H + W + 127) / 128, 128, 0, s>>>(TapAxis{Hin, y0, H, w, idx}, TapAxis{Win, x0, W, w + ny, idx + ny},
                                                scale, T);
  PRNU_CUDA_TRY(cudaGetLastError());
  k_fp_resize<<<dim3((W + 127) / 128, H), 128, 0, s>>>(K, pitch, w, idx, w + ny, idx + ny, T, H, W, out);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n += 2;
}
}  // namespace prnu

namespace prnu {
void launch_resid_scale(const double* partials, int nblk, int F, int H, int W, float* scale, cudaStream_t s,
                        LaunchCounter& lc) {
  k_resid_scale<<<F, 256, 0, s>>>(partials, nblk, H, W, scale);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}
void launch_fill(float* p, int n, float v, cudaStream_t s, LaunchCounter& lc) {
  k_fill<<<(n + 255) / 256, 256, 0, s>>>(p, n, v);
  PRNU_CUDA_TRY(cudaGetLastError());
  lc.n++;
}
}  // namespace prnu
