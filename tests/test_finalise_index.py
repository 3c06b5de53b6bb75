"""Index arithmetic of the finalisation (search_common.cuh), compiled for the
host: whatever the row statistics hold, the peak, the window's row pairs and
the rows that hold the parts of the energy lie inside the candidate's slot."""
import subprocess

import pytest

from paper_2207_14507_gb300 import buildlib

SOURCE = r"""
#include <stdio.h>
#include <vector>
#include "search_common.cuh"
using namespace prnu;

static FinPeak peak_of(const std::vector<RowStat>& st, int W) {
  float v = -INFINITY;
  int i = INT_MAX;
  for (size_t y = 0; y < st.size(); ++y) take_row(v, i, st[y], (int)y, W);
  return peak_at(v, i, W);
}
static int fail(const char* what, int H, int W, int py) {
  printf("%s: H %d W %d py %d\n", what, H, W, py);
  return 1;
}
int main() {
  // rows without an ordered value, and rows never written
  for (int H : {16, 256, 720, 1080, 2160, 4096})
    for (int W : {16, 256, 1280, 1920, 3840, 4096})
      for (int arg : {INT_MAX, INT_MIN, -1, W}) {
        std::vector<RowStat> st(H, RowStat{-INFINITY, arg, 0.0});
        FinPeak p = peak_of(st, W);
        if (p.py != 0 || p.px != 0 || p.peak != -INFINITY) return fail("no maximum", H, W, p.py);
        st[H - 1] = RowStat{-3.f, W - 1, 0.0};   // one row has a value
        p = peak_of(st, W);
        if (p.py != H - 1 || p.px != W - 1 || p.peak != -3.f) return fail("one row", H, W, p.py);
        st[H / 2] = RowStat{-3.f, 2, 0.0};       // a tie: the first in row-major order
        p = peak_of(st, W);
        if (p.py != H / 2 || p.px != 2) return fail("tie", H, W, p.py);
      }
  // every peak row: six row pairs cover the window, the parts' row pair is none of them
  for (int H = 16; H <= 4096; H += 2)
    for (int py = 0; py < H; ++py) {
      const int s = fin_scratch_row(py, H);
      if (s < 0 || s > H - 2 || (s & 1)) return fail("scratch row", H, 0, py);
      int covered = 0;
      for (int b = 0; b < kFinPairParts; ++b) {
        const int p = window_pair(py, b, H);
        if (p < 0 || p >= H / 2 || p == s / 2) return fail("window pair", H, 0, py);
        for (int q = 0; q < 2; ++q) covered += cdist(2 * p + q, py, H) <= kHalfWindow;
      }
      if (covered != 2 * kHalfWindow + 1) return fail("window rows", H, 0, py);
    }
  static_assert(kFinParts * sizeof(double) <= 2 * 8 * sizeof(float2), "the parts fit a row pair of 16 columns");
  printf("ok\n");
  return 0;
}
"""


def test_indices_stay_inside_the_slot(tmp_path):
    try:
        nvcc = buildlib.nvcc()
    except RuntimeError:
        pytest.skip("no nvcc")
    src, exe = tmp_path / "index.cu", tmp_path / "index"
    src.write_text(SOURCE)
    subprocess.run([nvcc, *buildlib.ARCH, *buildlib.FLAGS, "-I" + buildlib.CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
