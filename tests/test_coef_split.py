"""The float pairs of the stiffness rows (csrc/coef_split.h), on the host.

Each row must sum to zero exactly as pairs, and no entry may move by more
than half of the last place of the row's largest entry (2^-49 of its binade)
plus its own rounding; the matrices are the library's own cell matrices.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2407_02100_gb300", "csrc")

PROG = r'''
#include "coef_split.h"
#include "setup.h"
#include <cstdio>
using namespace gmg;
int main() {
  for (int k = 1; k <= 8; ++k) {
    std::vector<double> M, K;
    cell_matrices_1d(k, M, K);
    const int n = k + 1;
    std::vector<float> h, l;
    split_zero_sum_rows(K.data(), n, n, h, l);
    for (int r = 0; r < n; ++r) {
      double sum = 0, big = 0;
      for (int c = 0; c < n; ++c) big = std::fmax(big, std::fabs(K[r * n + c]));
      for (int c = 0; c < n; ++c) {
        const double q = (double)h[r * n + c] + (double)l[r * n + c];
        sum += q;  // multiples of one power of two, far below 2^53 of it: exact
        if (!(std::fabs(q - K[r * n + c]) <= std::ldexp(big, -48))) { std::printf("entry %d %d %d\n", k, r, c); return 1; }
        if (!(std::fabs(l[r * n + c]) <= std::ldexp(std::fabs(h[r * n + c]), -24))) { std::printf("pair %d %d %d\n", k, r, c); return 1; }
      }
      if (sum != 0.0) { std::printf("sum %d %d %g\n", k, r, sum); return 1; }
    }
  }
  std::printf("ok\n");
  return 0;
}
'''


def test_stiffness_rows_sum_to_zero_as_pairs(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "split.cpp", tmp_path / "split"
    src.write_text(PROG)
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", f"-I{CSRC}", "-I/usr/local/cuda/include", str(src),
                    os.path.join(CSRC, "setup.cpp"), "-o", str(exe)], check=True, capture_output=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0 and res.stdout == "ok\n", res.stdout
