// Line operations of the patch sweep on two patches at once (pair_arith.cuh):
// rows of the two-cell patch matrices and the mirror-symmetric fast-
// diagonalisation transforms (App. A.3), with coefficient tables of this
// translation unit, in the arithmetic PA that the including file chooses.  A
// coefficient is kept as broadcast pairs, (h, h, l, l) or (c, c), so that one
// constant-memory read gives it ready for use.
#pragma once
#include <vector>

#include "../../include/gmg.h"
#include "coef_split.h"
#include "pair_arith.cuh"

#ifndef GMG_PAIR_ARITH
#error "define GMG_PAIR_ARITH (PairDF or PairF32) before including pair_lines.cuh"
#endif

namespace gmg {
namespace {

using PA = GMG_PAIR_ARITH;

__host__ __device__ constexpr int pl_off_patch(int k) { return k <= 1 ? 0 : pl_off_patch(k - 1) + (2 * k - 3) * (2 * k - 1); }
__host__ __device__ constexpr int pl_off_t(int k) { return k <= 1 ? 0 : pl_off_t(k - 1) + (2 * k - 3) * (2 * k - 3); }

// two-cell patch matrices, rows = interior closure rows 1..2k-1, columns 0..2k
__constant__ PA::tab p_M[pl_off_patch(9)];
__constant__ PA::tab p_K[pl_off_patch(9)];
// the negated end columns of rows 0..2k-2 (column 0 up to the vertex row, 2k
// after it; on the vertex row both hold the same entry): M then K per row
__constant__ PA::tab p_E[2 * 64];
__host__ __device__ constexpr int pl_off_end(int k) { return 2 * (k - 1) * (k - 1); }  // 2 (1 + 3 + ... + (2k - 3))
// fast-diagonalisation eigenvectors (row = node, column = mode)
__constant__ PA::tab p_T[pl_off_t(9)];

__device__ __forceinline__ PA::coef pl_coef(const PA::tab& c) { return PA::coefficient(c); }

// The rows that belong to one cell of the two-cell matrices M_p (KIND 0) and
// K_p (KIND 1), on the cell's closure values x[q], q = 0 at the outer end and
// q = K at the vertex (Q0 = 1: the outer end is left out).  The second cell is
// the mirror image of the first (E[K-p][K-q] = E[p][q]), so one body serves
// both.  pl_cell_row: acc += (FIRST: =) row p = 1..K-1; pl_centre: the cell's
// part of the vertex row, whose vertex column (of both cells) is added with
// `vertex` only.
template <int K, int KIND, bool FIRST, int Q0>
__device__ __forceinline__ void pl_cell_row(int p, const PA::val (&x)[K + 1], PA::acc& acc) {
  constexpr int C = 2 * K + 1;
#pragma unroll
  for (int q = Q0; q <= K; ++q) {
    const int o = pl_off_patch(K) + (p - 1) * C + q;
    const PA::coef c = pl_coef(KIND == 0 ? p_M[o] : p_K[o]);
    if (FIRST && q == Q0) acc = PA::first(c, x[q]);
    else PA::add(acc, c, x[q]);
  }
}
template <int K, int KIND, int Q0>
__device__ __forceinline__ void pl_centre(bool vertex, const PA::val (&x)[K + 1], PA::acc& acc) {
  constexpr int C = 2 * K + 1;
#pragma unroll
  for (int q = Q0; q < K; ++q) {
    const int o = pl_off_patch(K) + (K - 1) * C + q;
    PA::add(acc, pl_coef(KIND == 0 ? p_M[o] : p_K[o]), x[q]);
  }
  if (vertex) {
    const int o = pl_off_patch(K) + (K - 1) * C + K;
    PA::add(acc, pl_coef(KIND == 0 ? p_M[o] : p_K[o]), x[K]);
  }
}

// The sums and differences of mirrored entries are normalised (three of the 11
// operations): left loose, a whole FD solve errs 17 % more than with them.
// forward transform y_i = sum_j T[j][i] x_j; emit(i, y_i) per output
template <int K, typename F>
__device__ __forceinline__ void pl_forward(const PA::val (&x)[2 * K - 1], F&& emit) {
  constexpr int M = 2 * K - 1, c = K - 1;
  PA::val sv[K], dv[K > 1 ? K - 1 : 1];
#pragma unroll
  for (int j = 0; j < c; ++j) {
    sv[j] = PA::sum(x[j], x[M - 1 - j]);
    dv[j] = PA::diff(x[j], x[M - 1 - j]);
  }
  sv[c] = x[c];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    PA::acc acc = PA::first(pl_coef(p_T[pl_off_t(K) + i]), sv[0]);
#pragma unroll
    for (int j = 1; j <= c; ++j) PA::add(acc, pl_coef(p_T[pl_off_t(K) + j * M + i]), sv[j]);
    emit(i, PA::value(acc));
  }
#pragma unroll
  for (int i = K; i < M; ++i) {
    PA::acc acc = PA::first(pl_coef(p_T[pl_off_t(K) + i]), dv[0]);
#pragma unroll
    for (int j = 1; j < c; ++j) PA::add(acc, pl_coef(p_T[pl_off_t(K) + j * M + i]), dv[j]);
    emit(i, PA::value(acc));
  }
}

// backward transform x_j = sum_i T[j][i] y_i; emit(j, x_j) per output
template <int K, typename F>
__device__ __forceinline__ void pl_backward(const PA::val (&y)[2 * K - 1], F&& emit) {
  constexpr int M = 2 * K - 1, c = K - 1;
#pragma unroll
  for (int j = 0; j < c; ++j) {
    PA::acc e = PA::first(pl_coef(p_T[pl_off_t(K) + j * M]), y[0]);
#pragma unroll
    for (int i = 1; i < K; ++i) PA::add(e, pl_coef(p_T[pl_off_t(K) + j * M + i]), y[i]);
    PA::acc o = PA::first(pl_coef(p_T[pl_off_t(K) + j * M + K]), y[K]);
#pragma unroll
    for (int i = K + 1; i < M; ++i) PA::add(o, pl_coef(p_T[pl_off_t(K) + j * M + i]), y[i]);
    const PA::val ev = PA::value(e), ov = PA::value(o);
    emit(j, PA::sum(ev, ov));
    emit(M - 1 - j, PA::diff(ev, ov));
  }
  PA::acc e = PA::first(pl_coef(p_T[pl_off_t(K) + c * M]), y[0]);
#pragma unroll
  for (int i = 1; i < K; ++i) PA::add(e, pl_coef(p_T[pl_off_t(K) + c * M + i]), y[i]);
  emit(c, PA::value(e));
}

// fills this translation unit's transform of degree k
inline int pl_upload_transform(int k, const double* That) {
  const int M = 2 * k - 1;
  std::vector<PA::tab> t(M * M);
  for (int i = 0; i < M * M; ++i) {
    float h, l;
    split_pair(That[i], h, l);
    PA::make_tab(t[i], That[i], h, l);
  }
  const size_t e = sizeof(PA::tab);
  return cudaMemcpyToSymbol(p_T, t.data(), t.size() * e, pl_off_t(k) * e) == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

// fills this translation unit's tables of degree k
inline int pl_upload(int k, const double* Mp, const double* Kp, const double* That) {
  const int C = 2 * k + 1, M = 2 * k - 1;
  std::vector<PA::tab> m(M * C), s(M * C), end(2 * M);
  std::vector<float> kh, kl;
  split_patch_stiffness(Kp, k, kh, kl);
  float h, l;
  for (int i = 0; i < M * C; ++i) {
    split_pair(Mp[i], h, l);
    PA::make_tab(m[i], Mp[i], h, l);
    PA::make_tab(s[i], Kp[i], kh[i], kl[i]);
  }
  for (int i = 0; i < M; ++i) {
    const int o = i * C + (i < k ? 0 : C - 1);
    split_pair(Mp[o], h, l);
    PA::make_tab(end[2 * i], -Mp[o], -h, -l);
    PA::make_tab(end[2 * i + 1], -Kp[o], -kh[o], -kl[o]);
  }
  const size_t e = sizeof(PA::tab);
  if (cudaMemcpyToSymbol(p_M, m.data(), m.size() * e, pl_off_patch(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(p_K, s.data(), s.size() * e, pl_off_patch(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(p_E, end.data(), end.size() * e, pl_off_end(k) * e) != cudaSuccess)
    return GMG_ERR_CUDA;
  return pl_upload_transform(k, That);
}

}  // namespace
}  // namespace gmg
