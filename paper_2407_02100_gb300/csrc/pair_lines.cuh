// Line operations of the patch sweep on two patches at once (pair_arith.cuh):
// rows of the two-cell patch matrices and the mirror-symmetric fast-
// diagonalisation transforms (App. A.3), with coefficient tables of this
// translation unit.  Every coefficient is kept as the four floats (h, h, l, l),
// so that a 16-byte constant-memory read gives both broadcast pairs.
#pragma once
#include <vector>

#include "../../include/gmg.h"
#include "coef_split.h"
#include "pair_arith.cuh"

namespace gmg {
namespace {

__host__ __device__ constexpr int pl_off_patch(int k) { return k <= 1 ? 0 : pl_off_patch(k - 1) + (2 * k - 3) * (2 * k - 1); }
__host__ __device__ constexpr int pl_off_t(int k) { return k <= 1 ? 0 : pl_off_t(k - 1) + (2 * k - 3) * (2 * k - 3); }

// two-cell patch matrices, rows = interior closure rows 1..2k-1, columns 0..2k
__constant__ float4 p_M[pl_off_patch(9)];
__constant__ float4 p_K[pl_off_patch(9)];
// the negated end columns of rows 0..2k-2 (column 0 up to the vertex row, 2k
// after it; on the vertex row both hold the same entry): M then K per row
__constant__ float4 p_E[2 * 64];
__host__ __device__ constexpr int pl_off_end(int k) { return 2 * (k - 1) * (k - 1); }  // 2 (1 + 3 + ... + (2k - 3))
// fast-diagonalisation eigenvectors (row = node, column = mode)
__constant__ float4 p_T[pl_off_t(9)];

__device__ __forceinline__ df2_coef pl_coef(const float4& c) {
  const ulonglong2 v = reinterpret_cast<const ulonglong2&>(c);
  return {{v.x}, {v.y}};
}

// The rows that belong to one cell of the two-cell matrices M_p (KIND 0) and
// K_p (KIND 1), on the cell's closure values x[q], q = 0 at the outer end and
// q = K at the vertex (Q0 = 1: the outer end is left out).  The second cell is
// the mirror image of the first (E[K-p][K-q] = E[p][q]), so one body serves
// both.  pl_cell_row: acc += (FIRST: =) row p = 1..K-1; pl_centre: the cell's
// part of the vertex row, whose vertex column (of both cells) is added with
// `vertex` only.
template <int K, int KIND, bool FIRST, int Q0>
__device__ __forceinline__ void pl_cell_row(int p, const df2 (&x)[K + 1], df2_acc& acc) {
  constexpr int C = 2 * K + 1;
#pragma unroll
  for (int q = Q0; q <= K; ++q) {
    const int o = pl_off_patch(K) + (p - 1) * C + q;
    const df2_coef c = pl_coef(KIND == 0 ? p_M[o] : p_K[o]);
    if (FIRST && q == Q0) acc = df2_acc_first(c, x[q]);
    else df2_acc_add(acc, c, x[q]);
  }
}
template <int K, int KIND, int Q0>
__device__ __forceinline__ void pl_centre(bool vertex, const df2 (&x)[K + 1], df2_acc& acc) {
  constexpr int C = 2 * K + 1;
#pragma unroll
  for (int q = Q0; q < K; ++q) {
    const int o = pl_off_patch(K) + (K - 1) * C + q;
    df2_acc_add(acc, pl_coef(KIND == 0 ? p_M[o] : p_K[o]), x[q]);
  }
  if (vertex) {
    const int o = pl_off_patch(K) + (K - 1) * C + K;
    df2_acc_add(acc, pl_coef(KIND == 0 ? p_M[o] : p_K[o]), x[K]);
  }
}

// The sums and differences of mirrored entries are normalised (three of the 11
// operations): left loose, a whole FD solve errs 17 % more than with them.
// forward transform y_i = sum_j T[j][i] x_j; emit(i, y_i) per output
template <int K, typename F>
__device__ __forceinline__ void pl_forward(const df2 (&x)[2 * K - 1], F&& emit) {
  constexpr int M = 2 * K - 1, c = K - 1;
  df2 sv[K], dv[K > 1 ? K - 1 : 1];
#pragma unroll
  for (int j = 0; j < c; ++j) {
    sv[j] = df2_add(x[j], x[M - 1 - j]);
    dv[j] = df2_sub(x[j], x[M - 1 - j]);
  }
  sv[c] = x[c];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    df2_acc acc = df2_acc_first(pl_coef(p_T[pl_off_t(K) + i]), sv[0]);
#pragma unroll
    for (int j = 1; j <= c; ++j) df2_acc_add(acc, pl_coef(p_T[pl_off_t(K) + j * M + i]), sv[j]);
    emit(i, df2_acc_value(acc));
  }
#pragma unroll
  for (int i = K; i < M; ++i) {
    df2_acc acc = df2_acc_first(pl_coef(p_T[pl_off_t(K) + i]), dv[0]);
#pragma unroll
    for (int j = 1; j < c; ++j) df2_acc_add(acc, pl_coef(p_T[pl_off_t(K) + j * M + i]), dv[j]);
    emit(i, df2_acc_value(acc));
  }
}

// backward transform x_j = sum_i T[j][i] y_i; emit(j, x_j) per output
template <int K, typename F>
__device__ __forceinline__ void pl_backward(const df2 (&y)[2 * K - 1], F&& emit) {
  constexpr int M = 2 * K - 1, c = K - 1;
#pragma unroll
  for (int j = 0; j < c; ++j) {
    df2_acc e = df2_acc_first(pl_coef(p_T[pl_off_t(K) + j * M]), y[0]);
#pragma unroll
    for (int i = 1; i < K; ++i) df2_acc_add(e, pl_coef(p_T[pl_off_t(K) + j * M + i]), y[i]);
    df2_acc o = df2_acc_first(pl_coef(p_T[pl_off_t(K) + j * M + K]), y[K]);
#pragma unroll
    for (int i = K + 1; i < M; ++i) df2_acc_add(o, pl_coef(p_T[pl_off_t(K) + j * M + i]), y[i]);
    const df2 ev = df2_acc_value(e), ov = df2_acc_value(o);
    emit(j, df2_add(ev, ov));
    emit(M - 1 - j, df2_sub(ev, ov));
  }
  df2_acc e = df2_acc_first(pl_coef(p_T[pl_off_t(K) + c * M]), y[0]);
#pragma unroll
  for (int i = 1; i < K; ++i) df2_acc_add(e, pl_coef(p_T[pl_off_t(K) + c * M + i]), y[i]);
  emit(c, df2_acc_value(e));
}

// fills this translation unit's tables of degree k
inline int pl_upload(int k, const double* Mp, const double* Kp, const double* That) {
  const int C = 2 * k + 1, M = 2 * k - 1;
  auto split = [](const double* a, int n) {
    std::vector<float4> t(n);
    for (int i = 0; i < n; ++i) {
      const float h = (float)a[i], l = (float)(a[i] - (double)h);
      t[i] = make_float4(h, h, l, l);
    }
    return t;
  };
  const std::vector<float4> m = split(Mp, M * C), t = split(That, M * M);
  std::vector<float> kh, kl;
  split_zero_sum_rows(Kp, M, C, kh, kl);
  std::vector<float4> s(M * C);
  for (int i = 0; i < M * C; ++i) s[i] = make_float4(kh[i], kh[i], kl[i], kl[i]);
  std::vector<float4> end(2 * M);
  for (int i = 0; i < M; ++i) {
    const float4 a = m[i * C + (i < k ? 0 : C - 1)], b = s[i * C + (i < k ? 0 : C - 1)];
    end[2 * i] = make_float4(-a.x, -a.y, -a.z, -a.w);
    end[2 * i + 1] = make_float4(-b.x, -b.y, -b.z, -b.w);
  }
  const size_t e = sizeof(float4);
  if (cudaMemcpyToSymbol(p_M, m.data(), m.size() * e, pl_off_patch(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(p_K, s.data(), s.size() * e, pl_off_patch(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(p_E, end.data(), end.size() * e, pl_off_end(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(p_T, t.data(), t.size() * e, pl_off_t(k) * e) != cudaSuccess)
    return GMG_ERR_CUDA;
  return GMG_OK;
}

}  // namespace
}  // namespace gmg
