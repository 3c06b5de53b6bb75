// fft_packed.cuh -- in-register DFTs for the kernels that hold a long
// butterfly (16 to 48 points) in one thread.
//
// A complex number is one packed FP32 pair: the add, mul and fma .f32x2
// instructions take two lanes per issue slot at the scalar instructions' lane
// rate (39.8 T lane-operations/s measured, scalar adds 39.1), so everything
// that treats the two parts alike takes half the issue slots.  Multiplications
// by +-i and by a complex constant mix the parts; they stay scalar, where
// swapping the pair would cost the moves it saves.  Every operation has its
// rounding fixed, so a transform gives the same bits in every kernel.
#pragma once
#include "fft.cuh"

namespace prnu {

__device__ __forceinline__ float2 p_add(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 p_sub(float2 a, float2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
// a * s and a * s + b, s real
__device__ __forceinline__ float2 p_scale(float2 a, float s) { return __fmul2_rn(a, make_float2(s, s)); }
__device__ __forceinline__ float2 p_axpy(float2 a, float s, float2 b) { return __ffma2_rn(a, make_float2(s, s), b); }
// a + q b, q = -i (forward) or +i (inverse)
template <bool INV>
__device__ __forceinline__ float2 p_add_quarter(float2 a, float2 b) {
  return INV ? make_float2(__fadd_rn(a.x, -b.y), __fadd_rn(a.y, b.x))
             : make_float2(__fadd_rn(a.x, b.y), __fadd_rn(a.y, -b.x));
}
// a + s q b, s real
template <bool INV>
__device__ __forceinline__ float2 p_axpy_quarter(float2 a, float s, float2 b) {
  return INV ? make_float2(__fmaf_rn(b.y, -s, a.x), __fmaf_rn(b.x, s, a.y))
             : make_float2(__fmaf_rn(b.y, s, a.x), __fmaf_rn(b.x, -s, a.y));
}
// v * w_N^M (see c_twiddle)
template <int M, int N, bool INV>
__device__ __forceinline__ float2 p_twiddle(float2 v) {
  constexpr int m = ((M % N) + N) % N;
  if constexpr (m == 0 || 2 * m == N || 4 * m == N || 4 * m == 3 * N) {
    return c_twiddle<M, N, INV>(v);
  } else {
    constexpr float c = float(ce_cos2pi(m, N));
    constexpr float s = float(INV ? ce_sin2pi(m, N) : -ce_sin2pi(m, N));
    return make_float2(__fmaf_rn(v.x, c, -__fmul_rn(v.y, s)), __fmaf_rn(v.x, s, __fmul_rn(v.y, c)));
  }
}

__host__ __device__ constexpr int ce_inv_mod(int a, int m) {   // 1/a modulo m
  for (int k = 1; k < m; ++k)
    if (a * k % m == 1) return k;
  return 1;
}
// the highest power in R of its smallest prime
__host__ __device__ constexpr int prime_power(int r) {
  int f = 1;
  for (int p = 2; p <= 5 && f == 1; ++p)
    while (r % p == 0) {
      r /= p;
      f *= p;
    }
  return f;
}

// X[k] = sum_n x[n] w_R^(nk) in place; products of coprime factors by Good's
// prime-factor map (no twiddles), prime powers by a Cooley-Tukey split.
template <int R, bool INV>
struct DftP {
  static constexpr int F = prime_power(R);
  static constexpr int P = F < R ? F : R % 4 == 0 && R > 8 ? 4 : R % 2 == 0 ? 2 : R % 3 == 0 ? 3 : 5;
  static constexpr int Q = R / P;
  static constexpr int UQ = F < R ? Q * ce_inv_mod(Q % P, P) : 1;   // output step of k1 and of k2
  static constexpr int UP = F < R ? P * ce_inv_mod(P % Q, Q) : P;

  template <int N2, int K1 = 0>
  __device__ __forceinline__ static void inner_twiddles(float2 (&t)[P]) {
    if constexpr (F == R && K1 < P) {
      t[K1] = p_twiddle<N2 * K1, R, INV>(t[K1]);
      inner_twiddles<N2, K1 + 1>(t);
    }
  }
  template <int N2 = 0>
  __device__ __forceinline__ static void first(const float2 (&x)[R], float2 (&y)[R]) {
    if constexpr (N2 < Q) {
      float2 t[P];
#pragma unroll
      for (int n1 = 0; n1 < P; ++n1) t[n1] = x[(Q * n1 + (F < R ? P : 1) * N2) % R];
      DftP<P, INV>::run(t);
      inner_twiddles<N2>(t);
#pragma unroll
      for (int k1 = 0; k1 < P; ++k1) y[k1 * Q + N2] = t[k1];
      first<N2 + 1>(x, y);
    }
  }
  __device__ __forceinline__ static void run(float2 (&x)[R]) {
    float2 y[R];
    first(x, y);
#pragma unroll
    for (int k1 = 0; k1 < P; ++k1) {
      float2 t[Q];
#pragma unroll
      for (int n2 = 0; n2 < Q; ++n2) t[n2] = y[k1 * Q + n2];
      DftP<Q, INV>::run(t);
#pragma unroll
      for (int k2 = 0; k2 < Q; ++k2) x[(k1 * UQ + k2 * UP) % R] = t[k2];
    }
  }
};

template <bool INV>
struct DftP<2, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[2]) {
    const float2 a = x[0], b = x[1];
    x[0] = p_add(a, b);
    x[1] = p_sub(a, b);
  }
};

template <bool INV>
struct DftP<3, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[3]) {
    constexpr float h = 0.8660254037844386f;   // sin(2 pi / 3)
    const float2 a = x[0], t = p_add(x[1], x[2]), u = p_sub(x[1], x[2]);
    const float2 m = p_axpy(t, -0.5f, a);
    x[0] = p_add(a, t);
    x[1] = p_axpy_quarter<INV>(m, h, u);
    x[2] = p_axpy_quarter<INV>(m, -h, u);
  }
};

template <bool INV>
struct DftP<4, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[4]) {
    const float2 s02 = p_add(x[0], x[2]), d02 = p_sub(x[0], x[2]);
    const float2 s13 = p_add(x[1], x[3]), d13 = p_sub(x[1], x[3]);
    x[0] = p_add(s02, s13);
    x[2] = p_sub(s02, s13);
    x[1] = p_add_quarter<INV>(d02, d13);
    x[3] = p_add_quarter<!INV>(d02, d13);
  }
};

template <bool INV>
struct DftP<5, INV> {
  __device__ __forceinline__ static void run(float2 (&x)[5]) {
    constexpr float c1 = float(ce_cos2pi(1, 5)), c2 = float(ce_cos2pi(2, 5));
    constexpr float s1 = float(ce_sin2pi(1, 5)), s2 = float(ce_sin2pi(2, 5));
    const float2 a = x[0];
    const float2 t1 = p_add(x[1], x[4]), t2 = p_add(x[2], x[3]);
    const float2 t3 = p_sub(x[1], x[4]), t4 = p_sub(x[2], x[3]);
    const float2 m1 = p_axpy(t2, c2, p_axpy(t1, c1, a)), m2 = p_axpy(t2, c1, p_axpy(t1, c2, a));
    const float2 n1 = p_axpy(t4, s2, p_scale(t3, s1)), n2 = p_axpy(t4, -s1, p_scale(t3, s2));
    x[0] = p_add(p_add(a, t1), t2);
    x[1] = p_add_quarter<INV>(m1, n1);   // forward: m1 - i n1
    x[4] = p_add_quarter<!INV>(m1, n1);
    x[2] = p_add_quarter<INV>(m2, n2);
    x[3] = p_add_quarter<!INV>(m2, n2);
  }
};

}  // namespace prnu
