// wavelet.cu -- noise residual by Mihcak's wavelet denoiser (the paper's
// denoiser, Sec. 2.2), as an alternative to the 3x3 Wiener residual.
//
// Per frame (FP32 throughout):
//   1. the frame, mirrored at its bottom and right edges up to multiples of
//      16 (Hp x Wp), as float;
//   2. four levels of the orthonormal separable transform with Daubechies'
//      8-tap filter, periodic: rows (low half | high half), then columns (low
//      half over high half), each level on the previous level's low-low
//      quadrant (the quadrant layout keeps every band at pitch Wp);
//   3. every detail coefficient c replaced by its noise part
//      c s0^2 / (s2 + s0^2), s2 = min over W in {3, 5, 7, 9} of
//      max(0, mean of c^2 over the W x W window of its band - s0^2), zeros
//      outside the band; the last low-low band replaced by 0;
//   4. the inverse transform of those noise parts: W(I) = I - F(I) (the
//      transform is linear), cropped to H x W; R = I W(I) or W(I).
// Two Hp x Wp buffers per frame.  Forward: the detail bands of every level in
// the quadrant layout (pitch Wp) in A, each level's low-low band, the next
// level's input, in T.  Then the noise parts in the quadrant layout in T, and
// the inverse's intermediate images in A; its last level goes straight to the
// residual.  Each level is one kernel each way: a block filters a tile along
// rows and columns through shared memory, two elements to a packed FP32
// instruction.
#include <algorithm>

#include "internal.h"

namespace prnu {

namespace {

// Daubechies' scaling filter with 4 vanishing moments, sum sqrt(2); wavelet
// filter g[k] = (-1)^k h[7 - k]
__host__ __device__ constexpr float wav_h(int k) {
  constexpr float h[8] = {0.2303778133088964f,  0.7148465705529154f,  0.6308807679298587f,
                          -0.0279837694168599f, -0.1870348117190931f, 0.0308413818355607f,
                          0.0328830116668852f,  -0.0105974017850690f};
  return h[k];
}
__host__ __device__ constexpr float wav_g(int k) { return (k & 1) ? -wav_h(7 - k) : wav_h(7 - k); }
// (value, value) or (a pair of coefficients) for the packed instructions
__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }

constexpr int kTS = 32;              // coefficients of a band per block and axis: 64 x 64 pixels
constexpr int kIn = 2 * kTS + 6;     // input samples of the analysis
constexpr int kPairs = kIn / 2;
constexpr int kBand = kTS + 3;       // coefficients of the synthesis
constexpr int kLevels = 4;

// a byte as a float: in the low mantissa bits of 2^23, minus 2^23
__device__ __forceinline__ float byte_float(uint32_t v) { return __uint_as_float(0x4B000000u | v) - 8388608.f; }

// elements i, i + 1 of out, i even and out aligned to the pair
template <int DT>
__device__ __forceinline__ void store_pair(void* out, size_t i, float a, float b) {
  if constexpr (DT == kF32) *reinterpret_cast<float2*>(reinterpret_cast<float*>(out) + i) = make_float2(a, b);
  else if constexpr (DT == kF16) *reinterpret_cast<__half2*>(reinterpret_cast<__half*>(out) + i) = __floats2half2_rn(a, b);
  else *reinterpret_cast<__nv_bfloat162*>(reinterpret_cast<__nv_bfloat16*>(out) + i) = __floats2bfloat162_rn(a, b);
}
__device__ __forceinline__ void copy4_async(float* dst, const float* src) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(__cvta_generic_to_global(src))
               : "memory");
}

// index i >= 0 of an axis of n samples, periodic
__device__ __forceinline__ int wrap_up(int i, int n) { return i < n ? i : i % n; }
// index i >= -3, periodic
__device__ __forceinline__ int wrap_both(int i, int n) { return i >= 0 ? wrap_up(i, n) : ((i % n) + n) % n; }
// sample i < 2 n of an axis of n samples, mirrored at its end (half-sample)
__device__ __forceinline__ int mirror(int i, int n) { return i < n ? i : 2 * n - 1 - i; }

// One level of the analysis: the h x w image (LEVEL0: the uint8 frame, mirrored
// to that size; else X, dense, of frame stride fstride) to its three detail
// bands in A (quadrant layout, pitch Wp) and, unless LL is null, its low-low
// band (dense h/2 x w/2).  A thread loads pairs of columns of pairs of rows, from
// one moving address where the tile holds no edge.  8 full-HD frames, all levels:
// 70 us (single samples, each with its edge tests: 84; a kernel per axis with 8
// global loads an output: 255); the first level, 38 of them, issues in 60% of
// cycles and uses 48% of the L1 pipe.
template <bool LEVEL0>
__global__ void __launch_bounds__(256) k_wav_analyse(const uint8_t* __restrict__ frames, size_t pitch, int H, int W,
                                                     const float* __restrict__ X, size_t fstride, int h, int w, int Wp,
                                                     float* __restrict__ A, float* __restrict__ LL) {
  __shared__ __align__(16) float2 in[kPairs * (kIn + 2)];   // (row 2p, row 2p + 1) at column x
  __shared__ float2 T[2][kPairs][kTS];                      // the same after the row filters, low and high
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int n0 = blockIdx.x * kTS, m0 = blockIdx.y * kTS, f = blockIdx.z;
  const int w2 = w / 2, h2 = h / 2;
  // row pair p, column pair c; LEVEL0 frames by byte pairs where these are aligned
  // and not mirrored
  const bool even = LEVEL0 && ((reinterpret_cast<uintptr_t>(frames) | pitch) & 1) == 0;
  auto pair = [&](int y, int x) -> float2 {
    if (!LEVEL0) return __ldg(reinterpret_cast<const float2*>(X + (size_t)f * fstride + (size_t)y * w + x));
    const uint8_t* row = frames + ((size_t)f * H + mirror(y, H)) * pitch;
    if (even && x + 1 < W) {
      const unsigned v = __ldg(reinterpret_cast<const uint16_t*>(row + x));
      return make_float2(byte_float(v & 255u), byte_float(v >> 8));
    }
    return make_float2(byte_float(__ldg(row + mirror(x, W))), byte_float(__ldg(row + mirror(x + 1, W))));
  };
  // no edge of the image inside the tile: one address, moved by constant steps
  const bool inner = 2 * m0 + kIn <= (LEVEL0 ? min(h, H) : h) && 2 * n0 + kIn <= (LEVEL0 ? min(w, W) : w) && (even || !LEVEL0);
  int p = threadIdx.x / kPairs, c = threadIdx.x - p * kPairs;
  const size_t pt = LEVEL0 ? pitch : (size_t)w;
  size_t at = (size_t)(2 * (m0 + p)) * pt + 2 * (n0 + c) + (LEVEL0 ? (size_t)f * H * pitch : (size_t)f * fstride);
#pragma unroll
  for (int e = 0; e < (kPairs * kPairs + 255) / 256; ++e) {
    if (p < kPairs) {
      float2 a, b;
      if (inner) {
        if (LEVEL0) {
          const unsigned va = __ldg(reinterpret_cast<const uint16_t*>(frames + at));
          const unsigned vb = __ldg(reinterpret_cast<const uint16_t*>(frames + at + pt));
          a = make_float2(byte_float(va & 255u), byte_float(va >> 8));
          b = make_float2(byte_float(vb & 255u), byte_float(vb >> 8));
        } else {
          a = __ldg(reinterpret_cast<const float2*>(X + at));
          b = __ldg(reinterpret_cast<const float2*>(X + at + pt));
        }
      } else {
        const int x = wrap_up(2 * (n0 + c), w);   // w is even: a pair does not wrap inside
        a = pair(wrap_up(2 * (m0 + p), h), x);
        b = pair(wrap_up(2 * (m0 + p) + 1, h), x);
      }
      *reinterpret_cast<float4*>(in + p * (kIn + 2) + 2 * c) = make_float4(a.x, b.x, a.y, b.y);
    }
    c += 256 % kPairs;
    p += 256 / kPairs;
    at += 2 * (256 / kPairs) * pt + 2 * (256 % kPairs);
    if (c >= kPairs) {
      c -= kPairs;
      ++p;
      at += 2 * pt - 2 * kPairs;
    }
  }
  __syncthreads();
  for (int p = wp; p < kPairs; p += 8) {
    const float4* src = reinterpret_cast<const float4*>(in + p * (kIn + 2)) + lane;
    float2 lo = dup(0.f), hi = dup(0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float4 v = src[j];
      const float2 a = make_float2(v.x, v.y), b = make_float2(v.z, v.w);
      lo = __ffma2_rn(a, dup(wav_h(2 * j)), lo);
      lo = __ffma2_rn(b, dup(wav_h(2 * j + 1)), lo);
      hi = __ffma2_rn(a, dup(wav_g(2 * j)), hi);
      hi = __ffma2_rn(b, dup(wav_g(2 * j + 1)), hi);
    }
    T[0][p][lane] = lo;
    T[1][p][lane] = hi;
  }
  __syncthreads();
  // columns: a warp takes the low or the high half, 8 output rows of each kind
  const int half = wp & 1, g = (wp >> 1) * 8, n = n0 + lane;
  if (n >= w2) return;
  float2 t[11];
#pragma unroll
  for (int i = 0; i < 11; ++i) t[i] = T[half][g + i][lane];
  const size_t fo = (size_t)f * fstride;
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const int m = m0 + g + k;
    if (m >= h2) break;
    float2 lo = dup(0.f), hi = dup(0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      lo = __ffma2_rn(t[k + j], make_float2(wav_h(2 * j), wav_h(2 * j + 1)), lo);
      hi = __ffma2_rn(t[k + j], make_float2(wav_g(2 * j), wav_g(2 * j + 1)), hi);
    }
    const float l = lo.x + lo.y, d = hi.x + hi.y;
    if (half) A[fo + (size_t)m * Wp + w2 + n] = l;
    else if (LL) LL[fo + (size_t)m * w2 + n] = l;
    A[fo + (size_t)(h2 + m) * Wp + (half ? w2 : 0) + n] = d;
  }
}

// Noise parts of the three detail bands of every level: band b of frame f,
// blockIdx.z = 3 f + b: 0 (rows high, columns low) at (0, w2), 1 at (h2, 0), 2 at
// (h2, w2) of a level of h2 x w2 coefficients a band; blockIdx.x counts the
// levels' tiles, finest level first.  Reads A, writes T.  The sums of c^2 over
// the 3, 5, 7 and 9 wide windows go along rows first (four sums a pixel, each a
// pair more than the last), then along columns.  The smallest of max(0, mean -
// s0) is max(0, smallest mean - s0): subtraction and max are monotone in
// floating point too.  A tile of 56 rows and its borders are 64, two whole
// turns of the row sums' lanes, and 7 rows of a column in a thread share the sums of
// two and of four rows that lie in several windows.  8 full-HD frames: 63 us, issue
// in 73% of cycles (tiles of 32 rows, 4 to a thread, each with its own sums: 121; 80
// shared loads a coefficient in a kernel per level: 211).
constexpr int kSX = 32, kSK = 7, kSY = 8 * kSK, kSR = 4;
// FAST: the quotients c s0 / den have no subnormal or overflowing part
template <bool FAST>
__global__ void __launch_bounds__(256) k_wav_shrink(const float* __restrict__ A, int Hp, int Wp, size_t fstride, float s0sq,
                                                    float* __restrict__ T) {
  // row pitches that put lanes of consecutive rows in distinct banks
  constexpr int SW = kSX + 2 * kSR + 4, SH = kSY + 2 * kSR, HW = kSX + 1;
  static_assert(SH == 64, "two rows a lane of the row sums");
  __shared__ __align__(16) float sq[SH * SW];
  __shared__ float2 ha[SH * HW], hb[SH * HW];   // (3, 5) and (7, 9) wide sums along rows
  const int f = blockIdx.z / 3, b = blockIdx.z - 3 * f;
  int h2 = Hp / 2, w2 = Wp / 2, tile = blockIdx.x, tx = (w2 + kSX - 1) / kSX, n = tx * ((h2 + kSY - 1) / kSY);
  while (tile >= n) {   // the level of this tile
    tile -= n;
    h2 /= 2;
    w2 /= 2;
    tx = (w2 + kSX - 1) / kSX;
    n = tx * ((h2 + kSY - 1) / kSY);
  }
  const int by0 = tile / tx * kSY, bx0 = (tile - tile / tx * tx) * kSX;
  const int oy = b == 0 ? 0 : h2, ox = b == 1 ? 0 : w2;
  const float* band = A + (size_t)f * fstride + (size_t)oy * Wp + ox;
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  {
    constexpr int C = kSX + 2 * kSR;
    static_assert(SH * C % 256 == 0, "whole steps of the block");
    int sy = threadIdx.x / C, sx = threadIdx.x - sy * C;
#pragma unroll
    for (int e = 0; e < SH * C / 256; ++e) {
      const int y = by0 + sy - kSR, x = bx0 + sx - kSR;
      float c = 0.f;
      if ((unsigned)y < (unsigned)h2 && (unsigned)x < (unsigned)w2) c = __ldg(band + (size_t)y * Wp + x);
      sq[sy * SW + sx] = c * c;
      sx += 256 % C;
      sy += 256 / C;
      if (sx >= C) {
        sx -= C;
        ++sy;
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < 2; ++q) {   // four adjacent pixels of a row, a lane per row
    const int sy = lane + 32 * q, x4 = wp * 4;
    const float4* p = reinterpret_cast<const float4*>(sq + sy * SW + x4);
    const float4 q0 = p[0], q1 = p[1], q2 = p[2];
    const float v[12] = {q0.x, q0.y, q0.z, q0.w, q1.x, q1.y, q1.z, q1.w, q2.x, q2.y, q2.z, q2.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float s1 = v[i + 3] + v[i + 4] + v[i + 5], s2 = s1 + (v[i + 2] + v[i + 6]);
      const float s3 = s2 + (v[i + 1] + v[i + 7]);
      ha[sy * HW + x4 + i] = make_float2(s1, s2);
      hb[sy * HW + x4 + i] = make_float2(s3, s3 + (v[i] + v[i + 8]));
    }
  }
  __syncthreads();
  const int x = bx0 + lane;
  if (x >= w2) return;
  // kSK adjacent rows of a column; sums of two and four rows are shared by the
  // rows whose windows hold them
  const int y0 = wp * kSK;
  float m[kSK];
  {
    const float2* src = ha + y0 * HW + lane;   // r[i] of row y0 + i - kSR
    float2 r[kSK + 2 * kSR], p[kSK + 2 * kSR];
#pragma unroll
    for (int i = 2; i < kSK + 6; ++i) r[i] = src[i * HW];
#pragma unroll
    for (int i = 2; i < kSK + 5; ++i) p[i] = __fadd2_rn(r[i], r[i + 1]);
#pragma unroll
    for (int k = 0; k < kSK; ++k) {
      const int i = k + kSR;
      m[k] = fminf((p[i - 1].x + r[i + 1].x) * (1.f / 9.f), (p[i - 2].y + p[i + 1].y + r[i].y) * (1.f / 25.f));
    }
  }
  {
    const float2* src = hb + y0 * HW + lane;
    float2 r[kSK + 2 * kSR], p[kSK + 2 * kSR], q[kSK + 2 * kSR];
#pragma unroll
    for (int i = 0; i < kSK + 8; ++i) r[i] = src[i * HW];
#pragma unroll
    for (int i = 0; i < kSK + 7; ++i) p[i] = __fadd2_rn(r[i], r[i + 1]);
#pragma unroll
    for (int i = 0; i < kSK + 5; ++i) q[i] = __fadd2_rn(p[i], p[i + 2]);
#pragma unroll
    for (int k = 0; k < kSK; ++k) {
      const int i = k + kSR;
      const float s7 = q[i - 3].x + (p[i + 1].x + r[i + 3].x), s9 = (q[i - 4].y + q[i].y) + r[i + 4].y;
      m[k] = fminf(m[k], fminf(s7 * (1.f / 49.f), s9 * (1.f / 81.f)));
    }
  }
  float* To = T + (size_t)f * fstride + (size_t)(oy + by0 + y0) * Wp + ox + x;
  const float* co = band + (size_t)(by0 + y0) * Wp + x;
#pragma unroll
  for (int k = 0; k < kSK; ++k) {
    if (by0 + y0 + k >= h2) break;
    const float c = __ldg(co + (size_t)k * Wp);
    const float den = fmaxf(m[k] - s0sq, 0.f) + s0sq, num = c * s0sq;
    float r;
    if (FAST) r = refined_quotient(num, den);
    else r = den > 0.f ? num / den : 0.f;
    To[(size_t)k * Wp] = r;
  }
}

// One level of the synthesis: the noise parts in D (quadrant layout, pitch Wp)
// and the low-low image LL (dense h/2 x w/2; null: zero) to the h x w image.
// OUT 0: dense into Y.  The last level: OUT 1 stores R = I W (or W) in `out`
// (dense [F][H][W]), OUT 2 the per-block sum of R^2 in partials, OUT 3
// R * scale[f].  8 full-HD frames, all levels: 79 us (loads through registers, a
// sample at a time: 104; a kernel per axis and one for the residual: 400), 51 of
// them in the last level, whose 66 MB of output HBM takes in 10.
template <int DT, int OUT>
__global__ void __launch_bounds__(256) k_wav_synth(const float* __restrict__ D, const float* __restrict__ LL, size_t fstride,
                                                   int h, int w, int Wp, float* __restrict__ Y,
                                                   const uint8_t* __restrict__ frames, size_t pitch, int H, int W, int f0,
                                                   int weight, void* __restrict__ out, double* __restrict__ partials,
                                                   const float* __restrict__ scale) {
  __shared__ __align__(16) float B[4][kBand][kTS + 4];         // the four bands, coefficient n at n - n0 + 3
  __shared__ __align__(16) float2 T[kTS][2][kTS + 4];          // (row 2i, row 2i + 1) after the column filters
  __shared__ double part[OUT == 2 ? kTS : 1];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int n0 = blockIdx.x * kTS, m0 = blockIdx.y * kTS, fl = blockIdx.z, f = f0 + fl;
  const int w2 = w / 2, h2 = h / 2;
  const size_t fo = (size_t)fl * fstride;
  {   // asynchronous copies: all of a thread's are in flight together
    constexpr int C = kTS + 4;
    const bool inner = m0 >= 3 && n0 >= 3 && m0 + kTS <= h2 && n0 + kTS < w2;   // no edge inside the tile
    int r = threadIdx.x / C, c = threadIdx.x - r * C;
    const float* d = D + fo + (size_t)max(m0 + r - 3, 0) * Wp + max(n0 + c - 3, 0);
    const float* ll = LL + fo + (size_t)max(m0 + r - 3, 0) * w2 + max(n0 + c - 3, 0);
    const size_t dh = (size_t)h2 * Wp;
#pragma unroll
    for (int e = 0; e < (kBand * C + 255) / 256; ++e) {
      if (r < kBand) {
        if (!inner) {
          const int m = wrap_both(m0 + r - 3, h2), n = wrap_both(n0 + c - 3, w2);
          d = D + fo + (size_t)m * Wp + n;
          ll = LL + fo + (size_t)m * w2 + n;
        }
        float* b = &B[0][0][0] + threadIdx.x + 256 * e;
        if (LL) copy4_async(b, ll);
        else *b = 0.f;
        copy4_async(b + kBand * C, d + dh);
        copy4_async(b + 2 * kBand * C, d + w2);
        copy4_async(b + 3 * kBand * C, d + dh + w2);
      }
      c += 256 % C;
      r += 256 / C;
      d += 256 / C * Wp + 256 % C;
      ll += 256 / C * w2 + 256 % C;
      if (c >= C) {
        c -= C;
        ++r;
        d += Wp - C;
        ll += w2 - C;
      }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
  }
  __syncthreads();
  // columns: outputs 2i and 2i + 1 take coefficients i - 3 .. i; a thread takes
  // two adjacent columns of the low or the high half, 5 values of i
  constexpr int kCP = (kTS + 4) / 2, kG = 5;
  if (threadIdx.x < 2 * kCP * 7) {
    const int q = threadIdx.x % (2 * kCP), g = threadIdx.x / (2 * kCP) * kG;
    const int half = q / kCP, c = (q - half * kCP) * 2;
    float2 lo[kG + 3], hi[kG + 3];
#pragma unroll
    for (int i = 0; i < kG + 3; ++i) {
      const int r = min(g + i, kBand - 1);
      lo[i] = *reinterpret_cast<const float2*>(&B[2 * half][r][c]);
      hi[i] = *reinterpret_cast<const float2*>(&B[2 * half + 1][r][c]);
    }
#pragma unroll
    for (int i = 0; i < kG; ++i) {
      if (g + i >= kTS) break;
      float2 a = dup(0.f), b = dup(0.f);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        a = __ffma2_rn(lo[i + 3 - j], dup(wav_h(2 * j)), a);
        a = __ffma2_rn(hi[i + 3 - j], dup(wav_g(2 * j)), a);
        b = __ffma2_rn(lo[i + 3 - j], dup(wav_h(2 * j + 1)), b);
        b = __ffma2_rn(hi[i + 3 - j], dup(wav_g(2 * j + 1)), b);
      }
      *reinterpret_cast<float4*>(&T[g + i][half][c]) = make_float4(a.x, b.x, a.y, b.y);
    }
  }
  __syncthreads();
  // rows: a warp takes a pair of rows, a lane outputs 2n and 2n + 1 of both
  const int x = 2 * (n0 + lane);
  const float s = OUT == 3 ? scale[f] : 1.f;
  const bool even_in = ((reinterpret_cast<uintptr_t>(frames) | pitch) & 1) == 0;
  const bool even_out = W % 2 == 0 && reinterpret_cast<uintptr_t>(out) % (DT == kF32 ? 8 : 4) == 0;
  float sq[kTS / 8] = {};   // R^2 over 2 x 2 pixels (OUT 2)
#pragma unroll
  for (int k = 0; k < kTS / 8; ++k) {
    const int i = wp + 8 * k, y = 2 * (m0 + i);
    if (OUT == 0 ? (y >= h || x >= w) : (y >= H || x >= W)) continue;
    float2 a = dup(0.f), b = dup(0.f);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 l = T[i][0][lane + 3 - j], d = T[i][1][lane + 3 - j];
      a = __ffma2_rn(l, dup(wav_h(2 * j)), a);
      a = __ffma2_rn(d, dup(wav_g(2 * j)), a);
      b = __ffma2_rn(l, dup(wav_h(2 * j + 1)), b);
      b = __ffma2_rn(d, dup(wav_g(2 * j + 1)), b);
    }
    if (OUT == 0) {
      *reinterpret_cast<float2*>(Y + fo + (size_t)y * w + x) = make_float2(a.x, b.x);
      *reinterpret_cast<float2*>(Y + fo + (size_t)(y + 1) * w + x) = make_float2(a.y, b.y);
    } else {
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        if (y + e >= H) break;
        float2 r = e ? make_float2(a.y, b.y) : make_float2(a.x, b.x);
        const bool two = x + 1 < W;
        if (weight) {
          const uint8_t* I = frames + ((size_t)f * H + y + e) * pitch + x;
          if (two && even_in) {
            const unsigned v = __ldg(reinterpret_cast<const uint16_t*>(I));
            r.x *= byte_float(v & 255u);
            r.y *= byte_float(v >> 8);
          } else {
            r.x *= byte_float(__ldg(I));
            r.y *= two ? byte_float(__ldg(I + 1)) : 0.f;
          }
        }
        if (OUT == 2) {
          sq[k] += fmaf(r.x, r.x, two ? r.y * r.y : 0.f);
        } else {
          const size_t o = ((size_t)f * H + y + e) * W + x;
          if (even_out) {
            store_pair<DT>(out, o, r.x * s, r.y * s);
          } else {
            store_store_type<DT>(out, o, r.x * s);
            if (two) store_store_type<DT>(out, o + 1, r.y * s);
          }
        }
      }
    }
  }
  if constexpr (OUT == 2) {   // float over a warp's two rows of 64 pixels, double beyond
    const double t = block_sum(sq, lane, wp, part);
    if (threadIdx.x == 0) partials[(size_t)f * gridDim.x * gridDim.y + blockIdx.y * gridDim.x + blockIdx.x] = t;
  }
}

int pad16(int n) { return (n + 15) / 16 * 16; }
dim3 tiles(int h, int w, int n) { return dim3((w / 2 + kTS - 1) / kTS, (h / 2 + kTS - 1) / kTS, n); }

}  // namespace

size_t wavelet_partials_needed(int F, int H, int W) {
  const dim3 g = tiles(pad16(H), pad16(W), 1);
  return (size_t)F * g.x * g.y;
}

void launch_wavelet_residual(const uint8_t* frames, int F, int H, int W, size_t pitch, int flags, int dtype,
                             float sigma0, void* out, float* scale, float* bufA, float* bufT, int chunk,
                             double* partials, cudaStream_t s, LaunchCounter& lc) {
  const int Hp = pad16(H), Wp = pad16(W);
  const size_t fs = (size_t)Hp * Wp;
  const int weight = (flags & PRNU_WEIGHT_BY_INTENSITY) ? 1 : 0;
  const bool norm = (flags & PRNU_NORMALISE) != 0;
  const float s0sq = sigma0 * sigma0;
  // offset of level l's dense image (l >= 1) in its buffer
  auto off = [&](int l) {
    size_t o = 0;
    for (int k = 1; k < l; ++k) o += (size_t)(Hp >> k) * (Wp >> k);
    return o;
  };
  const dim3 g0 = tiles(Hp, Wp, 1);
  const int nblk = (int)(g0.x * g0.y);
  ProfScope ps(lc, kKindResidual, s);
  for (int f0 = 0; f0 < F; f0 += chunk) {
    const int nf = std::min(chunk, F - f0);
    const uint8_t* fr = frames + (size_t)f0 * H * pitch;
    for (int l = 0; l < kLevels; ++l) {
      const int h = Hp >> l, w = Wp >> l;
      float* ll = l + 1 < kLevels ? bufT + off(l + 1) : nullptr;
      if (l == 0) k_wav_analyse<true><<<tiles(h, w, nf), 256, 0, s>>>(fr, pitch, H, W, nullptr, fs, h, w, Wp, bufA, ll);
      else k_wav_analyse<false><<<tiles(h, w, nf), 256, 0, s>>>(fr, pitch, H, W, bufT + off(l), fs, h, w, Wp, bufA, ll);
      PRNU_CUDA_TRY(cudaGetLastError());
    }
    unsigned ntiles = 0;
    for (int l = 0; l < kLevels; ++l)
      ntiles += (((Wp >> (l + 1)) + kSX - 1) / kSX) * (((Hp >> (l + 1)) + kSY - 1) / kSY);
    // |c| <= 16 * 255 (four levels of gain 2), so den <= 2^25 + s0 and c s0 <= 2^12 s0
    auto* shrink = s0sq >= 1e-18f && s0sq <= 1e18f ? k_wav_shrink<true> : k_wav_shrink<false>;
    shrink<<<dim3(ntiles, 1, 3 * nf), 256, 0, s>>>(bufA, Hp, Wp, fs, s0sq, bufT);
    PRNU_CUDA_TRY(cudaGetLastError());
    auto synth = [&](auto* fn, int l) {
      const int h = Hp >> l, w = Wp >> l;
      fn<<<tiles(h, w, nf), 256, 0, s>>>(bufT, l + 1 < kLevels ? bufA + off(l + 1) : nullptr, fs, h, w, Wp,
                                         l ? bufA + off(l) : nullptr, frames, pitch, H, W, f0, weight, out, partials, scale);
      PRNU_CUDA_TRY(cudaGetLastError());
      lc.n++;
    };
    for (int l = kLevels - 1; l >= 1; --l) synth(k_wav_synth<kF32, 0>, l);
    lc.n += kLevels + 1;
    if (!norm) {
      synth(dtype == kF32 ? k_wav_synth<kF32, 1> : dtype == kF16 ? k_wav_synth<kF16, 1> : k_wav_synth<kBF16, 1>, 0);
      continue;
    }
    // s = 1 / RMS(R) per frame, then the last level again with the scaled store
    synth(k_wav_synth<kF32, 2>, 0);
    launch_resid_scale(partials + (size_t)f0 * nblk, nblk, nf, H, W, scale + f0, s, lc);
    synth(dtype == kF32 ? k_wav_synth<kF32, 3> : dtype == kF16 ? k_wav_synth<kF16, 3> : k_wav_synth<kBF16, 3>, 0);
  }
  if (!norm && scale) launch_fill(scale, F, 1.f, s, lc);
}

}  // namespace prnu
