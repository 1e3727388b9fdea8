// Float pairs (hi, lo) of the coefficient matrices of the double-float kernels.
#pragma once
#include <algorithm>
#include <cmath>
#include <utility>
#include <vector>

namespace gmg {

inline void split_pair(double v, float& hi, float& lo) {
  hi = (float)v;
  lo = (float)(v - (double)hi);
}

// The rows of a stiffness matrix sum to zero (constants have no energy).
// Split entry by entry, the sums come out at the pairs' rounding, an error
// that a sweep repeats everywhere with the same sign and a V-cycle then
// amplifies.  So what a row of pairs is short of zero goes to its entries,
// largest first, each taking the multiple of its own last place (2^-48 of
// its binade) that comes nearest.  The largest entry takes up what the FP64
// row was short of zero itself and the rounding of every entry, at most
// (cols + 1) / 2 of its last places in all; any other moves by at most half of
// the last place of the next larger one and one of its own.  What is left is
// below the last place of the smallest.
inline void split_zero_sum_rows(const double* a, int rows, int cols, std::vector<float>& hi, std::vector<float>& lo) {
  hi.resize((size_t)rows * cols);
  lo.resize((size_t)rows * cols);
  std::vector<double> q(cols);
  std::vector<int> order(cols);
  for (int r = 0; r < rows; ++r) {
    const double* const row = a + (size_t)r * cols;
    for (int c = 0; c < cols; ++c) order[c] = c;
    std::sort(order.begin(), order.end(), [&](int x, int y) { return std::fabs(row[x]) > std::fabs(row[y]); });
    auto place = [&](int c) { return std::ldexp(1.0, std::ilogb(row[c]) - 48); };
    for (int c = 0; c < cols; ++c) q[c] = row[c] == 0.0 ? 0.0 : std::rint(row[c] / place(c)) * place(c);
    for (int i = 0; i < cols; ++i) {
      const int c = order[i];
      if (row[c] == 0.0) continue;
      long double sum = 0.0L;
      for (int j = 0; j < cols; ++j) sum += (long double)q[j];
      q[c] -= std::rint((double)sum / place(c)) * place(c);
    }
    for (int c = 0; c < cols; ++c) split_pair(q[c], hi[(size_t)r * cols + c], lo[(size_t)r * cols + c]);
  }
}

// The interior rows of the two-cell patch matrix Kp (2k - 1 rows, 2k + 1
// columns), as the sweeps read them: from the rows of the first cell alone, the
// second cell being its mirror image.  The vertex row is that cell's last row
// and its mirror image, which meet in the vertex entry, so it is split as the
// cell's row, with half of the vertex entry; corrected as one row of 2k + 1
// entries, mirrored ones would take different corrections, and the sum that is
// applied, twice the left half and the vertex, would not be zero (k = 8: -7e-14,
// -3e-14 split entry by entry).  What is split is the mean of the places where an
// entry of the cell's matrix stands (in either cell, transposed and mirrored): they
// differ by the rounding of the FP64 set-up, 5e-14 at k = 7, which the first cell's
// rows alone would pass on (error of a 3D Q7 sweep 3.2e-14, with the mean 2.8e-14).
inline void split_patch_stiffness(const double* Kp, int k, std::vector<float>& hi, std::vector<float>& lo) {
  const int C = 2 * k + 1, M = 2 * k - 1, n = k + 1;
  // entry (p, q), p >= 1, of the cell's matrix from both cells; half of the vertex entry
  auto entry = [&](int p, int q) {
    const double e = 0.5 * (Kp[(p - 1) * C + q] + Kp[(M - p) * C + 2 * k - q]);
    return p == k && q == k ? 0.5 * e : e;
  };
  std::vector<double> cell((size_t)k * n);  // rows 1..k
  for (int p = 1; p <= k; ++p)
    for (int q = 0; q < n; ++q) {
      double sum = 0.0;
      int places = 0;
      for (const auto& at : {std::pair<int, int>{p, q}, {q, p}, {k - p, k - q}, {k - q, k - p}})
        if (at.first >= 1) {  // (row 0 is the mirror image of row k)
          sum += entry(at.first, at.second);
          ++places;
        }
      cell[(size_t)(p - 1) * n + q] = sum / places;
    }
  std::vector<float> h, l;
  split_zero_sum_rows(cell.data(), k, n, h, l);
  hi.assign((size_t)M * C, 0.f);
  lo.assign((size_t)M * C, 0.f);
  for (int p = 0; p < k; ++p)
    for (int q = 0; q < n; ++q) {
      const float both = p == k - 1 && q == k ? 2.f : 1.f;  // the vertex entry, of both cells
      const int o = p * C + q;
      hi[o] = hi[M * C - 1 - o] = both * h[p * n + q];
      lo[o] = lo[M * C - 1 - o] = both * l[p * n + q];
    }
}

}  // namespace gmg
