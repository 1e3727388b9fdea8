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


# the sums of the two-cell rows as the two-patch kernels read them: a cell's
# row for either cell, the vertex row as twice its left half and the vertex
# entry, the end columns from the table of negated end entries.  Exact, in
# units of 2^-90.  No entry may move from the mean of its places by more than
# the header of coef_split.h says: half of the last place of the next larger one
# and one of its own, the largest by (k + 2) / 2 of its own, and what the FP64 row
# itself is short of zero.
PATCH = r'''
#include "coef_split.h"
#include "setup.h"
#include <cstdio>
using namespace gmg;
typedef __int128 I;
static I unit(float v) { return (I)std::ldexp((double)v, 90); }
int main() {
  for (int k = 1; k <= 8; ++k) {
    const int C = 2 * k + 1, M = 2 * k - 1;
    std::vector<double> Mp, Kp;
    assembled_1d(k, 2, 1, M, 0, C, Mp, Kp);
    std::vector<float> h, l;
    split_patch_stiffness(Kp.data(), k, h, l);
    auto pair = [&](int i, int c) { return unit(h[i * C + c]) + unit(l[i * C + c]); };
    for (int i = 0; i < k; ++i) {  // row i, from its left half
      I sum = 0;
      for (int c = 0; c <= k; ++c) sum += pair(i, c) * (i == k - 1 && c < k ? 2 : 1);
      if (sum != 0) { std::printf("sum %d %d %g\n", k, i, std::ldexp((double)sum, -90)); return 1; }
    }
    for (int i = 0; i < M; ++i) {
      I whole = 0;
      for (int c = 0; c < C; ++c) whole += pair(i, c);
      if (whole != 0) { std::printf("whole row %d %d\n", k, i); return 1; }
      for (int c = 0; c < C; ++c)
        if (h[i * C + c] != h[(M - 1 - i) * C + C - 1 - c] || l[i * C + c] != l[(M - 1 - i) * C + C - 1 - c]) {
          std::printf("mirror %d %d %d\n", k, i, c);
          return 1;
        }
    }
    for (int i = 0; i < k; ++i) {
      std::vector<double> row(k + 1);
      double defect = 0;
      // the cell's entry (r, c) in the first cell's rows, or the mirrored one in the second's
      auto at = [&](int r, int c) {
        const double half = r == k && c == k ? 0.5 : 1.0;
        return half * (Kp[(r - 1) * C + c] + Kp[(M - r) * C + 2 * k - c]) / 2;
      };
      for (int c = 0; c <= k; ++c) {
        const int r = i + 1, rs[4] = {r, c, k - r, k - c}, cs[4] = {c, r, k - c, k - r};
        double sum = 0;
        int n = 0;
        for (int j = 0; j < 4; ++j)
          if (rs[j] > 0) sum += at(rs[j], cs[j]), ++n;
        row[c] = sum / n;
        defect += row[c];
        if (!(std::fabs(row[c] - at(r, c)) <= 4e-15 * std::fabs(Kp[(k - 1) * C + k]))) { std::printf("mean %d %d %d\n", k, i, c); return 1; }
      }
      auto place = [&](double v) { return std::ldexp(1.0, std::ilogb(v) - 48); };
      for (int c = 0; c <= k; ++c) {
        double next = 0;  // the next larger entry (the mirror image on a middle row is as large)
        for (int d = 0; d <= k; ++d)
          if (std::fabs(row[d]) > std::fabs(row[c]) && (next == 0 || std::fabs(row[d]) < next)) next = std::fabs(row[d]);
        const double both = i == k - 1 && c == k ? 2.0 : 1.0;
        const double q = ((double)h[i * C + c] + (double)l[i * C + c]) / both;
        const double bound = next == 0 ? (k + 2) / 2.0 * place(row[c]) + std::fabs(defect) + 1e-15 * std::fabs(row[c])
                                       : place(next) / 2 + place(row[c]);
        if (!(std::fabs(q - row[c]) <= bound)) { std::printf("entry %d %d %d: %g above %g\n", k, i, c, q - row[c], bound); return 1; }
        if (!(std::fabs(l[i * C + c]) <= std::ldexp(std::fabs(h[i * C + c]), -24))) { std::printf("pair %d %d %d\n", k, i, c); return 1; }
      }
    }
  }
  std::printf("ok\n");
  return 0;
}
'''


def test_patch_rows_sum_to_zero_as_the_sweeps_read_them(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("needs g++")
    src, exe = tmp_path / "patch.cpp", tmp_path / "patch"
    src.write_text(PATCH)
    subprocess.run([gxx, "-std=c++17", "-O2", "-ffp-contract=off", f"-I{CSRC}", "-I/usr/local/cuda/include", str(src),
                    os.path.join(CSRC, "setup.cpp"), "-o", str(exe)], check=True, capture_output=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0 and res.stdout == "ok\n", res.stdout
