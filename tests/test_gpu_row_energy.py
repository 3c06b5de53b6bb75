"""Sums of squares of a row pair in the passes of sizes without planned kernels
(PairStat, row_generic.cuh): at most 8 plain FP32 terms a sum, then compensated
sums over a thread's sums and the warp."""
import subprocess

import pytest

from paper_2207_14507_gb300 import buildlib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <math.h>
#include <stdio.h>
#include <vector>
#include "row_generic.cuh"
using namespace prnu;

template <int R>
__global__ void rows(const float2* __restrict__ v, RowRed* __restrict__ out) {
  PairStat ps;
#pragma unroll
  for (int r = 0; r < R; ++r) ps.add(threadIdx.x + r * 32, r, v[threadIdx.x + r * 32]);
  const RowRed red = ps.reduce();
  if (threadIdx.x == 0) *out = red;
}

template <int R>
int check() {
  std::vector<float2> h(32 * R);
  unsigned z = 12345u + R;
  float2* d;
  RowRed *dr, r;
  if (cudaMalloc(&d, h.size() * sizeof(float2)) || cudaMalloc(&dr, sizeof(RowRed))) return printf("alloc\n");
  for (int test = 0; test < 2; ++test) {
    double ea = 0, eb = 0;
    for (int x = 0; x < 32 * R; ++x) {
      z = z * 1664525u + 1013904223u;
      const float u = (float)(z >> 8) / 16777216.f - 0.5f;
      // test 0: one square of 2^28 and ones, which a plain FP32 sum (units of 32) loses
      h[x] = test ? make_float2(u, 3.f * u * u) : make_float2(x == 0 ? 16384.f : x % 32 ? 1.f : 0.f, x % 32 == 5 ? 0.f : 1.f);
      ea += (double)h[x].x * h[x].x;
      eb += (double)h[x].y * h[x].y;
    }
    if (cudaMemcpy(d, h.data(), h.size() * sizeof(float2), cudaMemcpyHostToDevice)) return printf("copy\n");
    rows<R><<<1, 32>>>(d, dr);
    if (cudaMemcpy(&r, dr, sizeof(r), cudaMemcpyDeviceToHost)) return printf("run\n");
    const double ga = (double)r.sa + r.ca, gb = (double)r.sb + r.cb;
    const double tol = test ? 8 * ldexp(1.0, -24) : 0.0;   // 8 roundings of a sum of 8 terms; integers are exact
    if (fabs(ga - ea) > tol * ea || fabs(gb - eb) > tol * eb) return printf("R %d test %d: %.17g %.17g, %.17g %.17g\n", R, test, ga, ea, gb, eb);
    int ia = 0, ib = 0;
    for (int x = 1; x < 32 * R; ++x) {
      if (h[x].x > h[ia].x) ia = x;
      if (h[x].y > h[ib].y) ib = x;
    }
    if (r.ia != ia || r.ib != ib || r.ma != h[ia].x || r.mb != h[ib].y) return printf("R %d test %d: arg %d %d\n", R, test, r.ia, r.ib);
  }
  return 0;
}
int main() { return check<3>() || check<8>() || check<20>() || check<25>() || check<32>(); }
"""


def test_row_energies_against_double(tmp_path):
    src, exe = tmp_path / "rows.cu", tmp_path / "rows"
    src.write_text(SOURCE)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-I" + buildlib.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
