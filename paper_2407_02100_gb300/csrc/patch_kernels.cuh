// Pieces of the patch sweeps and the matrix-free operator kernels, templated on
// dimension and degree, for one scalar type GMG_T (this header is included once
// per type by patch_f64.cu / patch_f32.cu, each with its own __constant__
// tables).
//
// All level operators are written for unit-width cells: on a level with
// h = 1/n, A = h^{d-2} A_ref and A_j^{-1} = h^{2-d} A_ref,j^{-1}, so the
// coefficient tables do not depend on the level.
//
// Patch local_update (Sec. 3.1; Algorithm 4 runs it for every patch of one
// colour per launch; the sweeps are in pair_closure.cuh, face_kernels.cuh,
// pair_sweep_f64.cu, small_kernels.cuh and var_kernels.cuh):
//   gather    closure bar u_j ((2k+1)^d nodes) into shared memory
//   evaluate  r = h^{2-d} b_j - [A_ref bar u_j]_interior by sum factorisation
//             over the patch: the patch operator is a sum of tensor products
//             of the two-cell 1D matrices M_p, K_p (interior rows x closure
//             columns, banded: a row touches one cell, or two at the vertex)
//   solve     d = (T x .. x T) diag(1/sum lambda) (T x .. x T)^T r
//             (fast diagonalisation, App. A.3)
//   scatter   u_interior += omega d  (same-colour interiors are disjoint)
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "async.cuh"
#include "df_arith.cuh"
#include "kernels.h"

#ifndef GMG_T
#error "define GMG_T before including patch_kernels.cuh"
#endif

namespace gmg {
namespace GMG_NS {

using T = GMG_T;

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }
// compact per-degree offsets of the coefficient tables (degree k = 1..8)
__host__ __device__ constexpr int off_patch(int k) { return k <= 1 ? 0 : off_patch(k - 1) + (2 * k - 3) * (2 * k - 1); }
__host__ __device__ constexpr int off_t(int k) { return k <= 1 ? 0 : off_t(k - 1) + (2 * k - 3) * (2 * k - 3); }
__host__ __device__ constexpr int off_cell(int k) { return k <= 1 ? 0 : off_cell(k - 1) + k * k; }
constexpr int kPatchTotal = off_patch(9);
constexpr int kTTotal = off_t(9);
constexpr int kCellTotal = off_cell(9);

// two-cell patch matrices, rows = interior closure rows 1..2k-1, cols 0..2k
__constant__ T c_Mp[kPatchTotal];
__constant__ T c_Kp[kPatchTotal];
// fast-diagonalisation eigenvectors T[i][j] (row = node, column = mode)
__constant__ T c_T[kTTotal];
// unit-cell 1D mass and stiffness ((k+1)^2)
__constant__ T c_Mc[kCellTotal];
__constant__ T c_Kc[kCellTotal];
// the eigenvectors c_T split into float pairs hi + lo (double-float FD
// transforms of FP64 problems; unused by FP32 problems)
__constant__ float c_Thi[kTTotal];
__constant__ float c_Tlo[kTTotal];
// the two-cell patch matrices split the same way (double-float residual and
// face terms of FP64 problems)
__constant__ float c_Mphi[kPatchTotal];
__constant__ float c_Mplo[kPatchTotal];
__constant__ float c_Kphi[kPatchTotal];
__constant__ float c_Kplo[kPatchTotal];
// and the unit-cell matrices (double-float three-pass operator)
__constant__ float c_Mchi[kCellTotal];
__constant__ float c_Mclo[kCellTotal];
__constant__ float c_Kchi[kCellTotal];
__constant__ float c_Kclo[kCellTotal];

// band of closure row c (1..2k-1) of the two-cell patch matrices
__host__ __device__ constexpr int band_lo(int c, int K) { return c > K ? K : 0; }
__host__ __device__ constexpr int band_hi(int c, int K) { return c < K ? K : 2 * K; }


// acc + sign * sum_j E[i][j] x[j] over the band of closure row i+1 of the
// two-cell patch matrix E = M_p (KIND 0) or K_p (KIND 1); i = 0..M-1.  The
// __constant__ tables are indexed directly with compile-time offsets so that
// every coefficient is an immediate constant-bank operand.
template <int K, int KIND, bool NEG = false>
__device__ __forceinline__ T patch_row(int i, const T (&x)[2 * K + 1], T acc = T(0)) {
  constexpr int C = 2 * K + 1;
#pragma unroll
  for (int j = 0; j < C; ++j) {
    if (j >= band_lo(i + 1, K) && j <= band_hi(i + 1, K)) {
      const T e = KIND == 0 ? c_Mp[off_patch(K) + i * C + j] : c_Kp[off_patch(K) + i * C + j];
      acc = fma(NEG ? -e : e, x[j], acc);
    }
  }
  return acc;
}

// FD transforms of one line of M = 2K-1 values held in registers, using the
// mirror symmetry of the eigenvectors: modes 0..K-1 are even
// (T[M-1-j][i] = T[j][i]), modes K..M-1 odd (T[M-1-j][i] = -T[j][i]).
// forward: y_i = sum_j T[j][i] x_j;   backward: x_j = sum_i T[j][i] y_i
template <int K>
__device__ __forceinline__ void fd_forward(const T (&x)[2 * K - 1], T (&y)[2 * K - 1]) {
  constexpr int M = 2 * K - 1, c = K - 1;
    T sv[K], dv[K > 1 ? K - 1 : 1];
#pragma unroll
  for (int j = 0; j < c; ++j) {
    sv[j] = x[j] + x[M - 1 - j];
    dv[j] = x[j] - x[M - 1 - j];
  }
  sv[c] = x[c];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    T acc = T(0);
#pragma unroll
    for (int j = 0; j <= c; ++j) acc = fma(c_T[off_t(K) + j * M + i], sv[j], acc);
    y[i] = acc;
  }
#pragma unroll
  for (int i = K; i < M; ++i) {
    T acc = T(0);
#pragma unroll
    for (int j = 0; j < c; ++j) acc = fma(c_T[off_t(K) + j * M + i], dv[j], acc);
    y[i] = acc;
  }
}

template <int K>
__device__ __forceinline__ void fd_backward(const T (&y)[2 * K - 1], T (&x)[2 * K - 1]) {
  constexpr int M = 2 * K - 1, c = K - 1;
  #pragma unroll
  for (int j = 0; j < c; ++j) {
    T e = T(0), o = T(0);
#pragma unroll
    for (int i = 0; i < K; ++i) e = fma(c_T[off_t(K) + j * M + i], y[i], e);
#pragma unroll
    for (int i = K; i < M; ++i) o = fma(c_T[off_t(K) + j * M + i], y[i], o);
    x[j] = e + o;
    x[M - 1 - j] = e - o;
  }
  T e = T(0);
#pragma unroll
  for (int i = 0; i < K; ++i) e = fma(c_T[off_t(K) + c * M + i], y[i], e);
  x[c] = e;
}

// FD transform of a shared-memory line in place (stride s); with SCALE the
// result is multiplied elementwise by d[0], d[ds], ... (the diagonal).
template <int K, bool FORWARD, bool SCALE = false>
__device__ __forceinline__ void fd_smem_line(T* base, int s, const T* __restrict__ d = nullptr,
                                             int ds = 0) {
  constexpr int M = 2 * K - 1;
  T in[M], out[M];
#pragma unroll
  for (int j = 0; j < M; ++j) in[j] = base[j * s];
  if (FORWARD) fd_forward<K>(in, out);
  else fd_backward<K>(in, out);
#pragma unroll
  for (int j = 0; j < M; ++j) base[j * s] = SCALE ? out[j] * __ldg(d + j * ds) : out[j];
}

// The innermost transform pair of the FD solve on one shared-memory line
// (stride s) in registers: forward transform, times the diagonal d[0], d[ds],
// ..., backward transform.
template <int K>
__device__ __forceinline__ void fd_smem_line_solve(T* base, int s, const T* __restrict__ d, int ds) {
  constexpr int M = 2 * K - 1;
  T v[M], w[M];
#pragma unroll
  for (int j = 0; j < M; ++j) v[j] = base[j * s];
  fd_forward<K>(v, w);
#pragma unroll
  for (int j = 0; j < M; ++j) w[j] *= __ldg(d + j * ds);
  fd_backward<K>(w, v);
#pragma unroll
  for (int j = 0; j < M; ++j) base[j * s] = v[j];
}

// the FD transforms of fd_forward / fd_backward in double-float arithmetic
// (same mirror-symmetric even/odd splitting, eigenvectors from c_Thi/c_Tlo)
template <int K>
__device__ __forceinline__ void fd_forward_df(const dfv (&x)[2 * K - 1], dfv (&y)[2 * K - 1]) {
  constexpr int M = 2 * K - 1, c = K - 1;
  dfv sv[K], dv[K > 1 ? K - 1 : 1];
#pragma unroll
  for (int j = 0; j < c; ++j) {
    sv[j] = df_add(x[j], x[M - 1 - j]);
    dv[j] = df_add(x[j], df_neg(x[M - 1 - j]));
  }
  sv[c] = x[c];
#pragma unroll
  for (int i = 0; i < K; ++i) {
    df_acc acc = df_acc_first(c_Thi[off_t(K) + i], c_Tlo[off_t(K) + i], sv[0]);
#pragma unroll
    for (int j = 1; j <= c; ++j) df_acc_add(acc, c_Thi[off_t(K) + j * M + i], c_Tlo[off_t(K) + j * M + i], sv[j]);
    y[i] = df_acc_value(acc);
  }
#pragma unroll
  for (int i = K; i < M; ++i) {
    df_acc acc = df_acc_first(c_Thi[off_t(K) + i], c_Tlo[off_t(K) + i], dv[0]);
#pragma unroll
    for (int j = 1; j < c; ++j) df_acc_add(acc, c_Thi[off_t(K) + j * M + i], c_Tlo[off_t(K) + j * M + i], dv[j]);
    y[i] = df_acc_value(acc);
  }
}

template <int K>
__device__ __forceinline__ void fd_backward_df(const dfv (&y)[2 * K - 1], dfv (&x)[2 * K - 1]) {
  constexpr int M = 2 * K - 1, c = K - 1;
#pragma unroll
  for (int j = 0; j < c; ++j) {
    df_acc e = df_acc_first(c_Thi[off_t(K) + j * M], c_Tlo[off_t(K) + j * M], y[0]);
#pragma unroll
    for (int i = 1; i < K; ++i) df_acc_add(e, c_Thi[off_t(K) + j * M + i], c_Tlo[off_t(K) + j * M + i], y[i]);
    df_acc o = df_acc_first(c_Thi[off_t(K) + j * M + K], c_Tlo[off_t(K) + j * M + K], y[K]);
#pragma unroll
    for (int i = K + 1; i < M; ++i) df_acc_add(o, c_Thi[off_t(K) + j * M + i], c_Tlo[off_t(K) + j * M + i], y[i]);
    const dfv ev = df_acc_value(e), ov = df_acc_value(o);
    x[j] = df_add(ev, ov);
    x[M - 1 - j] = df_add(ev, df_neg(ov));
  }
  df_acc e = df_acc_first(c_Thi[off_t(K) + c * M], c_Tlo[off_t(K) + c * M], y[0]);
#pragma unroll
  for (int i = 1; i < K; ++i) df_acc_add(e, c_Thi[off_t(K) + c * M + i], c_Tlo[off_t(K) + c * M + i], y[i]);
  x[c] = df_acc_value(e);
}

// double-float FD transform of a shared-memory line (pairs, stride s) in place
template <int K, bool FORWARD>
__device__ __forceinline__ void fd_smem_line_df(float2* base, int s) {
  constexpr int M = 2 * K - 1;
  dfv in[M], out[M];
#pragma unroll
  for (int j = 0; j < M; ++j) {
    const float2 v = base[j * s];
    in[j] = {v.x, v.y};
  }
  if (FORWARD) fd_forward_df<K>(in, out);
  else fd_backward_df<K>(in, out);
#pragma unroll
  for (int j = 0; j < M; ++j) base[j * s] = make_float2(out[j].hi, out[j].lo);
}

// Shared-memory plan of a sweep kernel, per patch (elements):
//   IN  (NBUF copies): closure of u, then interior of b, rows of XU / XB
//       elements ([z][y][x]); with the TMA gather (TMA = true) a row is the
//       TMA box width: C (resp. M + 1) plus the alignment shift, rounded up to
//       16 bytes, and each box starts on 128 bytes
//   WA  3D: stage-y results A1, A2;  2D: stage-y results P, Q
//   WB  3D: stage-z results P, Q, then r and the FD work;  2D: r and FD work
// Stage x always reads WA and writes WB.
template <int DIM, int K, bool TMA = false>
struct SweepSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1;
  static constexpr int A = 16 / (int)sizeof(T);  // elements per 16 bytes
  static constexpr int XU = TMA ? (C + A - 1 + A - 1) / A * A : C;
  static constexpr int XB = TMA ? XU : M;
  static constexpr int R128 = 128 / (int)sizeof(T);
  static constexpr int rnd(int n) { return TMA ? (n + R128 - 1) / R128 * R128 : n; }
  static constexpr int NCLO = rnd(DIM == 3 ? C * C * XU : C * XU);
  static constexpr int NBIN = rnd(DIM == 3 ? M * M * XB : M * XB);
  static constexpr int NINT = DIM == 3 ? M * M * M : M * M;
  static constexpr int IN = NCLO + NBIN;
  static constexpr int WA = DIM == 3 ? 2 * C * M * M : 2 * C * M;
  static constexpr int WB = DIM == 3 ? cmax(2 * C * C * M, M * M * M) : M * M;
  static constexpr int per_patch(int nbuf) { return nbuf * IN + WA + WB; }
  // TMA box bytes of the closure of u and of the interior rows of b
  static constexpr int BOX_U = (DIM == 3 ? C * C * XU : C * XU) * (int)sizeof(T);
  static constexpr int BOX_B = (DIM == 3 ? M * M * XB : M * XB) * (int)sizeof(T);
};

// Tensor maps of the u and b vectors of each table entry (TMA gather).
template <int ME>
struct TmaMaps {
  CUtensorMap u[ME], b[ME];
};
template <>
struct TmaMaps<0> {};

// ---------------------------------------------------------------------------
// Matrix-free level operator on a tile of BC cells per direction.
// Global 1D matrix row for node i = c K + p: p > 0 -> cell c row p;
// p == 0 (vertex) -> cell c-1 row K plus cell c row 0.
// Tile inputs: nodes [(c0-1)K, (c0+BC)K] (EI per direction, zero outside the
// lattice); outputs: nodes [c0 K, (c0+BC) K) (EO per direction).
template <int K, int EI, int KIND>
__device__ __forceinline__ T cell_row(int o, const T (&x)[EI]) {
  // KIND 0: unit-cell mass, 1: unit-cell stiffness (direct __constant__ index)
  auto E = [](int i) -> T { return KIND == 0 ? c_Mc[off_cell(K) + i] : c_Kc[off_cell(K) + i]; };
  const int p = o % K;
  T acc = T(0);
  if (p == 0) {
#pragma unroll
    for (int q = 0; q <= K; ++q) acc = fma(E(K * (K + 1) + q), x[o + q], acc);
#pragma unroll
    for (int q = 0; q <= K; ++q) acc = fma(E(q), x[o + K + q], acc);
  } else {
#pragma unroll
    for (int q = 0; q <= K; ++q) acc = fma(E(p * (K + 1) + q), x[o - p + K + q], acc);
  }
  return acc;
}

// Tile of BX x BY (x BZ) cells: inputs E?I = (B? + 1) K + 1 nodes per
// direction (one halo cell below), outputs E?O = B? K.
template <int DIM, int K, int BX, int BY, int BZ>
struct ApplyDims {
  static constexpr int EIX = (BX + 1) * K + 1, EIY = (BY + 1) * K + 1, EIZ = DIM == 3 ? (BZ + 1) * K + 1 : 1;
  static constexpr int EOX = BX * K, EOY = BY * K, EOZ = DIM == 3 ? BZ * K : 1;
  // A: the input tile, later the stage-y results; B: the stage-z results
  static constexpr int SA = DIM == 3 ? cmax(EIX * EIY * EIZ, 2 * EIX * EOY * EOZ) : EIX * EIY;
  static constexpr int SB = DIM == 3 ? 2 * EIX * EIY * EOZ : 2 * EIX * EOY;
  static constexpr int SMEM_BYTES = (SA + SB) * (int)sizeof(T);
};

template <int DIM, int K, int BX, int BY, int BZ, int NT>
__global__ void __launch_bounds__(NT) apply_kernel(const T* __restrict__ xin, T* __restrict__ y,
                                                   const T* __restrict__ bvec, ApplyLaunch al) {
  using D = ApplyDims<DIM, K, BX, BY, BZ>;
  constexpr int EIX = D::EIX, EIY = D::EIY, EIZ = D::EIZ, EOX = D::EOX, EOY = D::EOY, EOZ = D::EOZ;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* A = reinterpret_cast<T*>(smem_raw);
  T* B = A + D::SA;
  const int N = al.g.N, n = al.g.n;
  const long long py = al.g.py, pz = al.g.pz;
  const int tx = (n + BX - 1) / BX, ty = (n + BY - 1) / BY, tz = DIM == 3 ? (n + BZ - 1) / BZ : 1;
  const int ntile = tx * ty * tz;
  const T alpha = (T)al.alpha, beta = (T)al.beta;

  for (int tid = blockIdx.x; tid < ntile; tid += gridDim.x) {
    const int t0 = tid % tx, t1 = (tid / tx) % ty, t2 = DIM == 3 ? tid / (tx * ty) : 0;
    const int g0 = (t0 * BX - 1) * K, g1 = (t1 * BY - 1) * K, g2 = DIM == 3 ? (t2 * BZ - 1) * K : 0;
    // gather the tile with zero fill outside the lattice
    const int nin = EIX * EIY * EIZ;
    for (int t = threadIdx.x; t < nin; t += NT) {
      int x = t % EIX, yy = (t / EIX) % EIY, z = DIM == 3 ? t / (EIX * EIY) : 0;
      int gx = g0 + x, gy = g1 + yy, gz = g2 + z;
      bool ok = gx >= 0 && gx < N && gy >= 0 && gy < N && (DIM == 2 || (gz >= 0 && gz < N));
      A[t] = ok ? xin[gx + py * gy + pz * gz] : T(0);
    }
    __syncthreads();
    if (DIM == 3) {
      // stage z: P = M_z x, Q = K_z x   (x:EIX, y:EIY, z:EOZ)
      for (int l = threadIdx.x; l < EIX * EIY; l += NT) {
        T v[EIZ];
#pragma unroll
        for (int j = 0; j < EIZ; ++j) v[j] = A[l + j * EIX * EIY];
#pragma unroll
        for (int o = 0; o < EOZ; ++o) {
          B[l + o * EIX * EIY] = cell_row<K, EIZ, 0>(o, v);
          B[EIX * EIY * EOZ + l + o * EIX * EIY] = cell_row<K, EIZ, 1>(o, v);
        }
      }
      __syncthreads();
      // stage y: A1 = M_y P, A2 = K_y P + M_y Q   (x:EIX, y:EOY, z:EOZ)
      for (int l = threadIdx.x; l < EIX * EOZ; l += NT) {
        int x0 = l % EIX, z = l / EIX;
        T p[EIY], q[EIY];
#pragma unroll
        for (int j = 0; j < EIY; ++j) {
          p[j] = B[x0 + j * EIX + z * EIX * EIY];
          q[j] = B[EIX * EIY * EOZ + x0 + j * EIX + z * EIX * EIY];
        }
#pragma unroll
        for (int o = 0; o < EOY; ++o) {
          A[x0 + o * EIX + z * EIX * EOY] = cell_row<K, EIY, 0>(o, p);
          A[EIX * EOY * EOZ + x0 + o * EIX + z * EIX * EOY] = cell_row<K, EIY, 1>(o, p) + cell_row<K, EIY, 0>(o, q);
        }
      }
      __syncthreads();
      // stage x and write: y = alpha (K_x A1 + M_x A2) + beta b on owned interior nodes
      for (int l = threadIdx.x; l < EOY * EOZ; l += NT) {
        int yy = l % EOY, z = l / EOY;
        int gy = g1 + K + yy, gz = g2 + K + z;
        if (gy <= 0 || gy >= N - 1 || gz <= 0 || gz >= N - 1) continue;
        T a1[EIX], a2[EIX];
#pragma unroll
        for (int j = 0; j < EIX; ++j) {
          a1[j] = A[j + EIX * (yy + EOY * z)];
          a2[j] = A[EIX * EOY * EOZ + j + EIX * (yy + EOY * z)];
        }
        const long long row = py * gy + pz * gz;
#pragma unroll
        for (int o = 0; o < EOX; ++o) {
          int gx = g0 + K + o;
          if (gx <= 0 || gx >= N - 1) continue;
          T v = alpha * (cell_row<K, EIX, 1>(o, a1) + cell_row<K, EIX, 0>(o, a2));
          if (bvec) v += beta * bvec[row + gx];
          y[row + gx] = v;
        }
      }
    } else {
      // one thread per line and cell: with a thread per line a tile kept 16
      // to 20 threads busy on chains of up to 100 FP64 operations
      // stage y: P = M_y x, Q = K_y x   (x:EIX, y:EOY)
      for (int t = threadIdx.x; t < EIX * BY; t += NT) {
        const int l = t % EIX, c = t / EIX;
        T v[2 * K + 1];
#pragma unroll
        for (int j = 0; j <= 2 * K; ++j) v[j] = A[l + (c * K + j) * EIX];
#pragma unroll
        for (int p = 0; p < K; ++p) {
          B[l + (c * K + p) * EIX] = cell_row<K, 2 * K + 1, 0>(p, v);
          B[EIX * EOY + l + (c * K + p) * EIX] = cell_row<K, 2 * K + 1, 1>(p, v);
        }
      }
      __syncthreads();
      // stage x and write
      for (int t = threadIdx.x; t < EOY * BX; t += NT) {
        const int c = t % BX, l = t / BX;
        const int gy = g1 + K + l;
        if (gy <= 0 || gy >= N - 1) continue;
        T p[2 * K + 1], q[2 * K + 1];
#pragma unroll
        for (int j = 0; j <= 2 * K; ++j) {
          p[j] = B[c * K + j + EIX * l];
          q[j] = B[EIX * EOY + c * K + j + EIX * l];
        }
        const long long row = py * gy;
#pragma unroll
        for (int o = 0; o < K; ++o) {
          const int gx = g0 + K + c * K + o;
          if (gx <= 0 || gx >= N - 1) continue;
          T v = alpha * (cell_row<K, 2 * K + 1, 1>(o, p) + cell_row<K, 2 * K + 1, 0>(o, q));
          if (bvec) v += beta * bvec[row + gx];
          y[row + gx] = v;
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace GMG_NS
}  // namespace gmg
