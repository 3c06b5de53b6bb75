// fft.cuh -- block-level mixed-radix FFT engine (device code).
//
// A length-n complex FFT (n = 2^a 3^b 5^c) runs in shared memory as a
// sequence of Stockham autosort stages (Govindaraju et al., SC'08 formulation):
// stage s with radix R and Ns = product of the previous radices reads, for
// butterfly j < n/R, the R inputs x[j + r*n/R], multiplies input r by
// w_{Ns*R}^{r*(j mod Ns)}, takes a length-R DFT in registers and writes output r
// to y[(j/Ns)*Ns*R + (j mod Ns) + r*Ns].
//
// The in-register DFTs of size R in {2,3,4,5,6,8,9,10,12,15,16} are built at
// compile time: sizes 2..5 from their closed forms, the others by a two-factor
// Cooley-Tukey split R = P*Q whose inner twiddles are compile-time constants.
// Those constants come from a constexpr Taylor series (they are only ever
// w_R^k for small R); the stage twiddles come from tables built in double
// precision and rounded to float.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>
#include <type_traits>

namespace prnu {

// ---------------------------------------------------------------- compile-time roots of unity

__host__ __device__ constexpr double ce_pi() { return 3.14159265358979323846264338327950288; }

// Taylor series, |x| <= pi/2 after reduction: 14 terms reach double rounding.
__host__ __device__ constexpr double ce_sin_poly(double x) {
  double term = x, sum = x;
  for (int k = 1; k < 14; ++k) {
    term *= -x * x / double((2 * k) * (2 * k + 1));
    sum += term;
  }
  return sum;
}
__host__ __device__ constexpr double ce_cos_poly(double x) {
  double term = 1.0, sum = 1.0;
  for (int k = 1; k < 14; ++k) {
    term *= -x * x / double((2 * k - 1) * (2 * k));
    sum += term;
  }
  return sum;
}
// cos and sin of 2*pi*m/n for integers m, n > 0.
__host__ __device__ constexpr double ce_cos2pi(long m, long n) {
  long r = ((m % n) + n) % n;
  if (2 * r > n) r -= n;                       // angle in (-pi, pi]
  double a = 2.0 * ce_pi() * double(r) / double(n);
  double aa = a < 0 ? -a : a;
  if (aa > ce_pi() / 2) return -ce_cos_poly(ce_pi() - aa);
  return ce_cos_poly(aa);
}
__host__ __device__ constexpr double ce_sin2pi(long m, long n) {
  long r = ((m % n) + n) % n;
  if (2 * r > n) r -= n;
  double a = 2.0 * ce_pi() * double(r) / double(n);
  double sg = a < 0 ? -1.0 : 1.0;
  double aa = a < 0 ? -a : a;
  if (aa > ce_pi() / 2) return sg * ce_sin_poly(ce_pi() - aa);
  return sg * ce_sin_poly(aa);
}

// ---------------------------------------------------------------- complex helpers

__device__ __forceinline__ float2 c_add(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 c_sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 c_mul(float2 a, float2 b) {
  return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
// a * conj(b)
__device__ __forceinline__ float2 c_mulc(float2 a, float2 b) {
  return make_float2(a.x * b.x + a.y * b.y, a.y * b.x - a.x * b.y);
}
__device__ __forceinline__ float2 c_conj(float2 a) { return make_float2(a.x, -a.y); }
// conj(a) * b with its rounding fixed: each component is one product rounded
// on its own plus one fused multiply-add, so every kernel that forms this
// product gets the same bits (no contraction left to the compiler's choice).
__device__ __forceinline__ float2 c_conj_mul(float2 a, float2 b) {
  return make_float2(__fmaf_rn(a.x, b.x, __fmul_rn(a.y, b.y)), __fmaf_rn(a.x, b.y, -__fmul_rn(a.y, b.x)));
}
// multiply by -i (forward quarter turn) / +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 c_quarter(float2 v) {
  return INV ? make_float2(-v.y, v.x) : make_float2(v.y, -v.x);
}

// v * w_N^M with w_N = exp(-2 pi i / N) (forward) or exp(+2 pi i / N) (inverse),
// M and N compile-time; exact quarter turns are done by swaps.
template <int M, int N, bool INV>
__device__ __forceinline__ float2 c_twiddle(float2 v) {
  constexpr int m = ((M % N) + N) % N;
  if constexpr (m == 0) {
    return v;
  } else if constexpr (2 * m == N) {
    return make_float2(-v.x, -v.y);
  } else if constexpr (4 * m == N) {
    return c_quarter<INV>(v);
  } else if constexpr (4 * m == 3 * N) {
    return c_quarter<!INV>(v);
  } else {
    constexpr float c = float(ce_cos2pi(m, N));
    constexpr float s = float(INV ? ce_sin2pi(m, N) : -ce_sin2pi(m, N));
    return make_float2(v.x * c - v.y * s, v.x * s + v.y * c);
  }
}

// ---------------------------------------------------------------- in-register DFTs

template <int R>
struct FirstFactor {
  static constexpr int value = (R % 4 == 0 && R != 4 && R != 8) ? 4 : (R % 2 == 0 ? 2 : (R % 3 == 0 ? 3 : 5));
};

template <int R, bool INV>
struct Dft;

template <bool INV>
struct Dft<2, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[2]) {
    float2 a = x[0], b = x[1];
    x[0] = c_add(a, b);
    x[1] = c_sub(a, b);
  }
};

template <bool INV>
struct Dft<3, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[3]) {
    constexpr float h = 0.8660254037844386f;  // sin(2 pi / 3)
    float2 a = x[0];
    float2 t = c_add(x[1], x[2]);
    float2 u = c_sub(x[1], x[2]);
    float2 m = make_float2(a.x - 0.5f * t.x, a.y - 0.5f * t.y);
    // forward: X1 = m - i h u, X2 = m + i h u
    float2 ihu = INV ? make_float2(-h * u.y, h * u.x) : make_float2(h * u.y, -h * u.x);
    x[0] = c_add(a, t);
    x[1] = c_add(m, ihu);
    x[2] = c_sub(m, ihu);
  }
};

template <bool INV>
struct Dft<4, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[4]) {
    float2 s02 = c_add(x[0], x[2]), d02 = c_sub(x[0], x[2]);
    float2 s13 = c_add(x[1], x[3]), d13 = c_quarter<INV>(c_sub(x[1], x[3]));
    x[0] = c_add(s02, s13);
    x[2] = c_sub(s02, s13);
    x[1] = c_add(d02, d13);
    x[3] = c_sub(d02, d13);
  }
};

template <bool INV>
struct Dft<5, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[5]) {
    constexpr float c1 = float(ce_cos2pi(1, 5)), c2 = float(ce_cos2pi(2, 5));
    constexpr float s1 = float(ce_sin2pi(1, 5)), s2 = float(ce_sin2pi(2, 5));
    float2 a = x[0];
    float2 t1 = c_add(x[1], x[4]), t2 = c_add(x[2], x[3]);
    float2 t3 = c_sub(x[1], x[4]), t4 = c_sub(x[2], x[3]);
    float2 m1 = make_float2(a.x + c1 * t1.x + c2 * t2.x, a.y + c1 * t1.y + c2 * t2.y);
    float2 m2 = make_float2(a.x + c2 * t1.x + c1 * t2.x, a.y + c2 * t1.y + c1 * t2.y);
    float2 n1 = make_float2(s1 * t3.x + s2 * t4.x, s1 * t3.y + s2 * t4.y);
    float2 n2 = make_float2(s2 * t3.x - s1 * t4.x, s2 * t3.y - s1 * t4.y);
    // forward: X1 = m1 - i n1, X4 = m1 + i n1, X2 = m2 - i n2, X3 = m2 + i n2
    float2 q1 = c_quarter<INV>(n1), q2 = c_quarter<INV>(n2);
    x[0] = make_float2(a.x + t1.x + t2.x, a.y + t1.y + t2.y);
    x[1] = c_add(m1, q1);
    x[4] = c_sub(m1, q1);
    x[2] = c_add(m2, q2);
    x[3] = c_sub(m2, q2);
  }
};

// Composite R = P*Q: n = Q*n1 + n2, k = k1 + P*k2;
// X[k1 + P k2] = sum_n2 w_Q^{n2 k2} w_R^{n2 k1} sum_n1 x[Q n1 + n2] w_P^{n1 k1}.
// The compile-time index loops are forced-inline template recursions so that
// every array stays in registers.
template <int R, bool INV, int P, int N2, int K1>
struct CompTwiddle {
  __device__ __forceinline__ static void run(const float2 (&t)[P], float2 (&y)[R]) {
    if constexpr (K1 < P) {
      y[N2 * P + K1] = c_twiddle<N2 * K1, R, INV>(t[K1]);
      CompTwiddle<R, INV, P, N2, K1 + 1>::run(t, y);
    }
  }
};

template <int R, bool INV, int P, int Q, int N2>
struct CompInner {
  __device__ __forceinline__ static void run(const float2 (&x)[R], float2 (&y)[R]) {
    if constexpr (N2 < Q) {
      float2 t[P];
#pragma unroll
      for (int n1 = 0; n1 < P; ++n1) t[n1] = x[Q * n1 + N2];
      Dft<P, INV>::run(t);
      CompTwiddle<R, INV, P, N2, 0>::run(t, y);
      CompInner<R, INV, P, Q, N2 + 1>::run(x, y);
    }
  }
};

template <int R, bool INV>
struct Dft {
  static constexpr int P = FirstFactor<R>::value;
  static constexpr int Q = R / P;
  __device__ __forceinline__ static void run(float2 (&x)[R]) {
    float2 y[R];
    CompInner<R, INV, P, Q, 0>::run(x, y);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) {
      float2 t[Q];
#pragma unroll
      for (int n2 = 0; n2 < Q; ++n2) t[n2] = y[n2 * P + k1];
      Dft<Q, INV>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) x[k1 + P * k2] = t[k2];
    }
  }
};

// ---------------------------------------------------------------- plans

constexpr int kMaxStages = 8;
constexpr int kMaxFft = 4096;

// A length-n plan: radices in execution order; per stage the product of the
// earlier radices, ceil(2^32 / ns) (j mod ns by one high multiplication, exact
// for j < 2^16) and the place of its twiddles in the plan's table tab
// (fft_plan.cuh), in float4.  ra, rb: where n is the product of two radices that one thread can
// hold, the two-stage plan of the column pass (col_generic.cuh), with the
// twiddles of its second forward and second inverse stage; else 0.  r3: where
// one thread cannot hold radices of such a plan in few registers, the row
// passes' three radices (row_generic.cuh), w3 the twiddles of the second and
// third stage, inv3 the reciprocal of r3[0]; else 0.
struct FftPlan {
  const float4* tab;
  int n;
  int nstages;
  int radix[kMaxStages];
  int ns[kMaxStages];
  unsigned inv[kMaxStages];
  int tw[kMaxStages];
  int min_radix;
  int ra, rb, tw_fwd, tw_inv;
  int r3[3], w3[2];
  unsigned inv3;
};

// float4 entries of a stage's twiddles
__host__ __device__ constexpr int stage_tw_len(int R, int ns) { return ns > 1 ? (R / 2) * ns : 0; }

}  // namespace prnu
