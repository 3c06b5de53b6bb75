"""block_sum (common.cuh): plain FP32 over the 32 lanes that hold one value, double
beyond, for each count of values a thread that the kernels use."""
import subprocess

import pytest

from paper_2207_14507_gb300 import buildlib

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <math.h>
#include <stdio.h>
#include <vector>
#include "common.cuh"
using namespace prnu;

template <int N>
__global__ void total(const float* __restrict__ in, double* __restrict__ out) {
  __shared__ double part[8 * N];
  float v[N];
#pragma unroll
  for (int k = 0; k < N; ++k) v[k] = in[k * 256 + threadIdx.x];
  const double t = block_sum(v, threadIdx.x & 31, threadIdx.x >> 5, part);
  if (threadIdx.x == 0) *out = t;
}

template <int N>
int check() {
  std::vector<float> h(256 * N);
  float* d;
  double *dout, got;
  if (cudaMalloc(&d, h.size() * sizeof(float)) || cudaMalloc(&dout, sizeof(double))) return printf("alloc\n");
  for (int test = 0; test < 3; ++test) {
    double want = 0;
    for (size_t i = 0; i < h.size(); ++i) {
      // distinct integers; ones beside a 2^24, which loses only those of its 32 lanes; random
      h[i] = test == 0 ? (float)(i * i % 1021) : test == 1 ? (i == 256 * (N - 1) + 37 ? 16777216.f : 1.f) : sinf((float)i) + 1.f;
      want += h[i];
    }
    if (cudaMemcpy(d, h.data(), h.size() * sizeof(float), cudaMemcpyHostToDevice)) return printf("copy\n");
    total<N><<<1, 256>>>(d, dout);
    if (cudaMemcpy(&got, dout, sizeof(got), cudaMemcpyDeviceToHost)) return printf("run\n");
    const double tol = test == 0 ? 0.0 : test == 1 ? 32.0 : 5 * ldexp(want, -24);
    if (!(fabs(got - want) <= tol)) return printf("N %d test %d: %.17g %.17g\n", N, test, got, want);
  }
  return 0;
}
int main() { return check<1>() || check<2>() || check<4>() || check<8>() || check<16>() || check<32>(); }
"""


def test_block_sums_against_double(tmp_path):
    src, exe = tmp_path / "sums.cu", tmp_path / "sums"
    src.write_text(SOURCE)
    subprocess.run([buildlib.nvcc(), *buildlib.ARCH, *buildlib.FLAGS, "-I" + buildlib.CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout
