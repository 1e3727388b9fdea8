// Float pairs (hi, lo) of the coefficient matrices of the double-float kernels.
#pragma once
#include <algorithm>
#include <cmath>
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
// its binade) that comes nearest: no entry moves by more than half of the
// last place of the next larger one, and what is left is below the last
// place of the smallest.
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

}  // namespace gmg
