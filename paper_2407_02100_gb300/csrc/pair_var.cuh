// Variable-coefficient patch sweep (degree <= 3), PA::W patches per thread
// (pair_arith.cuh: two in FP32, one in FP64), for the arithmetic PA of the
// including file; patches without a learned correction (those with one take
// patch_var_kernel).
//
// One colour of Algorithm 4: the local residual is evaluated cell by cell
// with the cell coefficients (Sec. 3.1, eq. "main:4"), the local solver is the
// fast diagonalisation of the constant-coefficient patch scaled by theta /
// abar (geometric mean and damping of the patch's coefficients):
//   u += omega theta / abar FD_ref(h^{2-d} b - sum_c a_c A_c u)
// The 2^d cells of a patch are contracted together: a line of the closure
// gives the K rows of either of its two cells (the vertex row in both,
// unsummed), so that a contraction serves the cells on both sides of the
// other axes, and only the last one, which knows its cell, multiplies by a_c.
// That takes half of the multiplications of 2^d separate cell operators.
#pragma once
#include <algorithm>
#include <type_traits>

#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "kernels.h"
#include "pair_lines.cuh"

namespace gmg {
namespace {

using T = PA::T;
using V = PA::val;
using E = PA::mem;
constexpr bool DF = sizeof(T) == 8;

// unit-cell matrices, rows 1..k, columns 0..k (the second cell is the mirror
// image of the first)
constexpr int kVarDegree = 3;
__host__ __device__ constexpr int v_off(int k) { return k <= 1 ? 0 : v_off(k - 1) + (k - 1) * k; }
__constant__ PA::tab v_M[v_off(kVarDegree + 1)];
__constant__ PA::tab v_K[v_off(kVarDegree + 1)];

template <int K, int KIND, bool FIRST>
__device__ __forceinline__ void var_row(int p, const V (&x)[K + 1], PA::acc& acc) {
#pragma unroll
  for (int q = 0; q <= K; ++q) {
    const int o = v_off(K) + (p - 1) * (K + 1) + q;
    const PA::coef c = pl_coef(KIND == 0 ? v_M[o] : v_K[o]);
    if (FIRST && q == 0) acc = PA::first(c, x[q]);
    else PA::add(acc, c, x[q]);
  }
}

// Shared memory per pair (one patch in FP64): the two fields of a contraction, [z][y][x] with 2k
// rows per contracted axis; stages work in place.  u and b go from global
// memory straight to registers (lanes along x): without room for them twice
// as many CTAs fit on an SM, which overlap one another's loads and barriers.
template <int DIM, int K>
struct VarSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1, H = 2 * K;
  static constexpr int NINT = DIM == 3 ? M * M * M : M * M;
  static constexpr int R = DIM == 3 ? C : H;             // row (x)
  static constexpr int F = DIM == 3 ? C * H * R : C * R;  // one field
  static constexpr int NCELL = 1 << DIM;
  static constexpr int bytes(int pp) { return pp * (2 * F + NCELL) * (int)sizeof(E); }
};

struct VarArgs {
  PatchLaunch pl;
  T* u;
  const T* b;
  const T* coef;
  const T* vscale;  // abar, theta per interior vertex
  const T* dinv;
};

// A CTA takes W PP consecutive patches of the colour, a thread the same line
// of patches 2q and 2q + 1 (W = 2).  Stages, 3D (2D: without the first, and y for z):
//   y: P, Q (on -u), 2k rows | x: A1, A2, 2k rows each way |
//   z: a_c (K_z A1 + M_z A2) per column of a cell pair |
//   z: r = h^{2-d} b + the columns of a node (1, 2 or 4), forward transform |
//   y: forward | x: forward, diagonal, backward | y: backward |
//   z: backward, u += omega theta / abar d
template <int DIM, int K, int NT, int PP, int CTAS, bool PRE>
__global__ void __launch_bounds__(NT, CTAS) pair_var_kernel(const __grid_constant__ VarArgs va) {
  using Z = VarSmem<DIM, K>;
  constexpr int C = Z::C, M = Z::M, H = Z::H, R = Z::R, F = Z::F, W = PA::W, NP = W * PP;
  constexpr int LINES = DIM == 3 ? M * M : M, NCELL = Z::NCELL;
  static_assert(NP <= NT, "one thread sets up one patch");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  E* const S = reinterpret_cast<E*>(smem_raw);  // [PP][2][F]
  E* const CO = S + PP * 2 * F;                  // [PP][NCELL] cell coefficients of both patches
  __shared__ long long s_origin[NP], s_cell[NP];
  __shared__ T s_scale[NP];
  const PatchLaunch& pl = va.pl;
  const long long py = pl.g.py, pz = pl.g.pz;
  const int g0 = blockIdx.x * NP, nv = min(NP, pl.n_patches - g0), npair = (nv + W - 1) / W, n = pl.g.n;
  const float sb = (float)pl.sb;  // an integer power of the cell count, exact in float
  if ((int)threadIdx.x < NP) {  // (a lone last patch is carried twice and stored once)
    const int q = threadIdx.x, pid = g0 + min(q, nv - 1);
    const int i0 = pid % pl.count[0], rest = pid / pl.count[0];
    const int i1 = rest % pl.count[1], i2 = DIM == 3 ? rest / pl.count[1] : 0;
    const int v0 = pl.first[0] + 2 * i0, v1 = pl.first[1] + 2 * i1, v2 = DIM == 3 ? pl.first[2] + 2 * i2 : 1;
    s_origin[q] = (v0 - 1) * K + py * ((v1 - 1) * K) + (DIM == 3 ? pz * ((v2 - 1) * K) : 0);
    s_cell[q] = (v0 - 1) + (long long)n * ((v1 - 1) + (DIM == 3 ? (long long)n * (v2 - 1) : 0));
    const long long vid = (v0 - 1) + (long long)(n - 1) * ((v1 - 1) + (DIM == 3 ? (long long)(n - 1) * (v2 - 1) : 0));
    s_scale[q] = (T)pl.omega * va.vscale[2 * vid + 1] / va.vscale[2 * vid];
  }
  __syncthreads();
  for (int t = threadIdx.x; t < npair * NCELL; t += NT) {
    const int q = t / NCELL, c = t % NCELL;
    const long long o = (c & 1) + (long long)n * (((c >> 1) & 1) + (DIM == 3 ? (long long)n * (c >> 2) : 0));
    PA::store(CO[t], PA::pack(va.coef[s_cell[W * q] + o], va.coef[s_cell[W * q + W - 1] + o]));
  }
  // the rows of b are on their way from the start
  constexpr bool EARLY = PRE && PP * LINES <= NT;
  const long long ps = DIM == 3 ? pz : py;
  T eb[EARLY ? 2 * M : 1];
  auto rhs = [&](int t, int p) -> const T* {
    const int ln = t % LINES;
    return va.b + s_origin[W * (t / LINES) + p] + 1 + ln % M + (DIM == 3 ? py * (1 + ln / M) : 0) + ps;
  };
  if constexpr (EARLY) {
    const int t = (int)threadIdx.x < npair * LINES ? threadIdx.x : 0;
#pragma unroll
    for (int l = 0; l < M; ++l) {
      eb[l] = __ldg(rhs(t, 0) + ps * l);
      eb[M + l] = __ldg(rhs(t, W - 1) + ps * l);
    }
  }
  // row of a cell-wise axis that holds interior node i (the first of the two
  // at the vertex)
  auto pos = [](int i) { return i + (i >= K ? 1 : 0); };
  auto line_rows = [&](auto&& get, auto&& put) {  // put(row, M v, K v)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      V v[K + 1];
#pragma unroll
      for (int q = 0; q <= K; ++q) v[q] = get(r ? 2 * K - q : q);
#pragma unroll
      for (int p = 1; p <= K; ++p) {
        PA::acc m, k;
        var_row<K, 0, true>(p, v, m);
        var_row<K, 1, true>(p, v, k);
        put(r ? 2 * K - p : p - 1, PA::value(m), PA::value(k));
      }
    }
  };

  if (DIM == 3) {
    // ---- y: P = M_y u, Q = K_y u on lines (x, z), from -u ----
    for (int t = threadIdx.x; t < npair * C * C; t += NT) {
      const int q = t / (C * C), x = t % C, z = t % (C * C) / C;
      const T *const a = va.u + s_origin[W * q] + x + pz * z, *const b = va.u + s_origin[W * q + W - 1] + x + pz * z;
      E* const P = S + q * 2 * F + z * H * R + x;
      line_rows([&](int y) -> V { return PA::pack_neg(a[py * y], b[py * y]); },
                [&](int j, V m, V k) {
                  PA::store(P[j * R], m);
                  PA::store(P[F + j * R], k);
                });
    }
    __syncthreads();
    // ---- x: A1 = M_x P, A2 = K_x P + M_x Q on rows (y, z), in place ----
    for (int t = threadIdx.x; t < npair * C * H; t += NT) {
      E* const P = S + t / (C * H) * 2 * F + t % (C * H) * R;
      V a1[H], a2[H];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        V v[K + 1], w[K + 1];
#pragma unroll
        for (int q = 0; q <= K; ++q) {
          v[q] = PA::load(P[r ? 2 * K - q : q]);
          w[q] = PA::load(P[F + (r ? 2 * K - q : q)]);
        }
#pragma unroll
        for (int p = 1; p <= K; ++p) {
          PA::acc m, k;
          var_row<K, 0, true>(p, v, m);
          var_row<K, 1, true>(p, v, k);
          var_row<K, 0, false>(p, w, k);
          a1[r ? 2 * K - p : p - 1] = PA::value(m);
          a2[r ? 2 * K - p : p - 1] = PA::value(k);
        }
      }
#pragma unroll
      for (int i = 0; i < H; ++i) {
        PA::store(P[i], a1[i]);
        PA::store(P[F + i], a2[i]);
      }
    }
  } else {
    // ---- x: P = M_x u, Q = K_x u on rows y, from -u ----
    for (int t = threadIdx.x; t < npair * C; t += NT) {
      const int q = t / C, y = t % C;
      const T *const a = va.u + s_origin[W * q] + py * y, *const b = va.u + s_origin[W * q + W - 1] + py * y;
      E* const P = S + q * 2 * F + y * R;
      line_rows([&](int x) -> V { return PA::pack_neg(a[x], b[x]); },
                [&](int i, V m, V k) {
                  PA::store(P[i], m);
                  PA::store(P[F + i], k);
                });
    }
  }
  __syncthreads();
  // ---- slowest axis: the weighted column of the cells (ox, oy, 0 and 1),
  // one value per interior node, in place of the first field ----
  constexpr int SL = DIM == 3 ? H * R : R;  // stride of the slowest axis
  constexpr int COLS = DIM == 3 ? H * H : H;
  for (int t = threadIdx.x; t < npair * COLS; t += NT) {
    const int q = t / COLS, X = t % COLS % H, Y = t % COLS / H;
    const int c = (X >= K ? 1 : 0) + (DIM == 3 && Y >= K ? 2 : 0);  // cell of the column at the low end
    constexpr int UP = DIM == 3 ? 4 : 2;                             // and at the high end: c + UP
    E* const P = S + q * 2 * F + (DIM == 3 ? Y * R : 0) + X;
    PA::acc col[M];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const PA::coef a = PA::weight(CO[q * NCELL + c + (r ? UP : 0)]);
      V v[K + 1], w[K + 1];
#pragma unroll
      for (int s = 0; s <= K; ++s) {
        v[s] = PA::load(P[(r ? 2 * K - s : s) * SL]);
        w[s] = PA::load(P[F + (r ? 2 * K - s : s) * SL]);
      }
#pragma unroll
      for (int p = 1; p <= K; ++p) {
        PA::acc acc;
        var_row<K, 1, true>(p, v, acc);
        var_row<K, 0, false>(p, w, acc);
        const int l = r ? 2 * K - p - 1 : p - 1;
        if (r == 1 && p == K) PA::add(col[l], a, PA::value(acc));
        else col[l] = PA::first(a, PA::value(acc));
      }
    }
#pragma unroll
    for (int l = 0; l < M; ++l) PA::store(P[l * SL], PA::value(col[l]));
  }
  __syncthreads();
  // ---- r = h^{2-d} b + the columns of each node, forward transform ----
  auto column = [&](int q, int ln) -> E* {
    return S + q * 2 * F + (DIM == 3 ? pos(ln / M) * R + pos(ln % M) : pos(ln));
  };
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES, i = ln % M, j = ln / M;
    const T *const ba = rhs(t, 0), *const bb = rhs(t, W - 1);
    E* const w = column(q, ln);
    const bool two_x = i == K - 1, two_y = DIM == 3 && j == K - 1;
    V r[M];
#pragma unroll
    for (int l = 0; l < M; ++l) {
      V s = PA::load(w[l * SL]);
      if (two_x) s = PA::sum(s, PA::load(w[l * SL + 1]));
      if (two_y) {
        V s2 = PA::load(w[l * SL + R]);
        if (two_x) s2 = PA::sum(s2, PA::load(w[l * SL + R + 1]));
        s = PA::sum(s, s2);
      }
      V rb;
      if constexpr (EARLY) rb = PA::pack(eb[l], eb[M + l]);
      else rb = PA::pack(__ldg(ba + ps * l), __ldg(bb + ps * l));
      r[l] = PA::sum(PA::value(PA::scaled(sb, rb)), s);
    }
    pl_forward<K>(r, [&](int l, V v) { PA::store(w[l * SL], v); });
  }
  __syncthreads();
  // ---- local solve by fast diagonalisation (App. A.3), in place ----
  auto line_y = [&](auto forward) {
    for (int t = threadIdx.x; t < npair * LINES; t += NT) {
      const int q = t / LINES, ln = t % LINES;  // x + M z
      E* const w = S + q * 2 * F + ln / M * SL + pos(ln % M);
      V v[M];
#pragma unroll
      for (int j = 0; j < M; ++j) v[j] = PA::load(w[pos(j) * R]);
      auto put = [&](int j, V x) { PA::store(w[pos(j) * R], x); };
      if constexpr (decltype(forward)::value) pl_forward<K>(v, put);
      else pl_backward<K>(v, put);
    }
    __syncthreads();
  };
  if (DIM == 3) line_y(std::true_type());
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;  // 3D: y + M z; 2D: y
    E* const w = S + q * 2 * F + (DIM == 3 ? ln / M * SL + pos(ln % M) * R : ln * SL);
    V v[M], x[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = PA::load(w[pos(i)]);
    // (the diagonal is symmetric in its indices)
    pl_forward<K>(v, [&](int i, V y) { x[i] = PA::diagonal(va.dinv, Z::NINT, i * LINES + ln, y); });
    pl_backward<K>(x, [&](int i, V y) { PA::store(w[pos(i)], y); });
  }
  __syncthreads();
  if (DIM == 3) line_y(std::false_type());
  // ---- backward along the slowest axis and scatter ----
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;
    const E* const w = column(q, ln);
    V v[M];
#pragma unroll
    for (int l = 0; l < M; ++l) v[l] = PA::load(w[l * SL]);
    const bool two = W == 2 && 2 * q + 1 < nv;
    const int x = 1 + ln % M, y = DIM == 3 ? 1 + ln / M : 0;
    const long long ofs = x + (DIM == 3 ? py * y : 0) + ps;
    T *const ga = va.u + s_origin[W * q] + ofs, *const gb = va.u + s_origin[W * q + W - 1] + ofs;
    const T sa = s_scale[W * q], sc = s_scale[W * q + W - 1];
    T oa[M], ob[M];
#pragma unroll
    for (int l = 0; l < M; ++l) {
      oa[l] = ga[ps * l];
      ob[l] = gb[ps * l];
    }
    pl_backward<K>(v, [&](int l, V d) {
      ga[ps * l] = fma(sa, PA::x(d), oa[l]);
      if (two) gb[ps * l] = fma(sc, PA::y(d), ob[l]);
    });
  }
}

// ---- host side ----

template <int DIM, int K, int NT, int PP, int CTAS, bool PRE>
int var_pair_launch(const PatchLaunch& pl, T* u, const T* b, const T* coef, const T* vscale, const T* dinv,
                    cudaStream_t s) {
  if (pl.n_patches <= 0) return GMG_OK;
  constexpr int SMEM = VarSmem<DIM, K>::bytes(PP);
  static_assert(SMEM <= 227 * 1024, "sweep kernel shared memory exceeds the per-CTA limit");
  auto kern = pair_var_kernel<DIM, K, NT, PP, CTAS, PRE>;
  static PerDevice<bool> ready_dev;  // attribute set once per device
  bool* const ready = ready_dev.get();
  if (!ready) return GMG_ERR_CUDA;
  if (!*ready) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess)
      return GMG_ERR_CUDA;
    *ready = true;
  }
  const VarArgs va{pl, u, b, coef, vscale, dinv};
  kern<<<(pl.n_patches + PA::W * PP - 1) / (PA::W * PP), NT, SMEM, s>>>(va);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

// Shapes: patches (FP32: pairs) and threads per CTA, and the CTAs per SM that the
// registers are limited for (0: left to the compiler); PRE: the rows of b are
// loaded before the first stage.  Up to LIMIT patches as many as fill the threads
// with the lines of the first stage, above it the shape of a full chip.
//
// FP64 takes one patch per thread: two were slower at every size, and twice as
// slow as one patch per CTA on small colours.  Per sweep (us), one patch per CTA -> two
// per thread -> now: 3D Q3 16^3 99 -> 197 -> 99, 24^3 205 -> 197 -> 123, 64^3 3479
// -> 1364 -> 1193; Q2 16^3 81 -> 131 -> 66, 64^3 1688 -> 361 -> 323; Q1 16^3 49 ->
// 89 -> 49, 64^3 600 -> 115 -> 82; 2D Q3 80^2 41 -> 62 -> 33, 640^2 1555 -> 291 ->
// 233.  Shapes at 3D Q3 64^3: 10 in 256 threads 1209, 5 in 256 1309 (16^3: 135, 98),
// 5 in 128 1390, limited for 2 CTAs 1588; Q2 64^3 14 in 128 331, 5 in 128 382 (16^3:
// 114, 68).  Colours that leave an SM to each patch last as long as one patch
// takes, and patch_var_kernel, whose threads share a patch cell by cell, is the
// shortest there: 3D Q3 8^3 82 us against 98, Q2 66 against 74 (16^3: 99, 98), 2D Q3
// 4^2 33 against 37.
//
// FP32, two patches per thread: 3D Q3 16^3 65 -> 49 with the small shape (2 pairs in
// 128 threads; 24^3 66 both), Q2 16^3 66 -> 49 (64^3: 129, 131), Q1 32^3 65 -> 49; Q3
// 64^3 5 in 128 317, 1 in 32 341.
template <int DIM, int K>
struct VarPairCfg {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1, LINES = DIM == 3 ? M * M : M, FIRST = DIM == 3 ? C * C : C;
  static constexpr bool PRE = DF || DIM == 2;
  // a full chip
  static constexpr int NT = DF && DIM == 3 && K == 3 ? 256 : 128;
  static constexpr int PP = DF && (DIM == 2 || K == 1) ? NT / FIRST : std::max(1, std::min(NT / LINES, 3 * NT / 8));
  static constexpr int CTAS = DF ? 0 : 1;
  // small colours
  static constexpr int SPP = DF ? NT / FIRST : K == 1 ? 3 : K == 2 ? 5 : 2, SNT = !DF && K == 1 ? 32 : NT;
  static constexpr int LIMIT = DIM == 2 ? 0 : DF ? (K == 1 ? 0 : 8000) : K == 3 ? 2000 : 8000;
  static constexpr int ONE = DF && K >= (DIM == 3 ? 2 : 3) ? 152 : 0;  // patch_var_kernel: the SMs of the chip
};

template <int DIM, int K>
int var_pair_impl(const PatchLaunch& pl, T* u, const T* b, const T* coef, const T* vscale, const T* dinv,
                  cudaStream_t s) {
  using Cfg = VarPairCfg<DIM, K>;
  if (pl.n_patches <= Cfg::ONE) return launch_patch_var<T>(pl, u, b, coef, vscale, dinv, nullptr, 0, s);
  if constexpr (Cfg::LIMIT > 0) {
    if (pl.n_patches <= Cfg::LIMIT)
      return var_pair_launch<DIM, K, Cfg::SNT, Cfg::SPP, 0, Cfg::PRE>(pl, u, b, coef, vscale, dinv, s);
  }
  return var_pair_launch<DIM, K, Cfg::NT, Cfg::PP, Cfg::CTAS, Cfg::PRE>(pl, u, b, coef, vscale, dinv, s);
}

}  // namespace

template <>
int upload_var_pair_tables<T>(int k, const double* Mc, const double* Kc, const double* That) {
  if (k < 1 || k > kVarDegree) return GMG_OK;
  const int n = k + 1;
  std::vector<PA::tab> m(k * n), s(k * n);
  std::vector<float> kh, kl;
  split_zero_sum_rows(Kc, n, n, kh, kl);
  for (int p = 1; p <= k; ++p)
    for (int q = 0; q <= k; ++q) {
      float h, l;
      split_pair(Mc[p * n + q], h, l);
      PA::make_tab(m[(p - 1) * n + q], Mc[p * n + q], h, l);
      PA::make_tab(s[(p - 1) * n + q], Kc[p * n + q], kh[p * n + q], kl[p * n + q]);
    }
  const size_t e = sizeof(PA::tab);
  if (cudaMemcpyToSymbol(v_M, m.data(), m.size() * e, v_off(k) * e) != cudaSuccess ||
      cudaMemcpyToSymbol(v_K, s.data(), s.size() * e, v_off(k) * e) != cudaSuccess)
    return GMG_ERR_CUDA;
  return pl_upload_transform(k, That);
}

template <>
int launch_patch_var_pair<T>(const PatchLaunch& pl, T* u, const T* b, const T* coef, const T* vscale, const T* dinv,
                             cudaStream_t s) {
  switch (pl.g.dim * 16 + pl.g.k) {
    case 2 * 16 + 1: return var_pair_impl<2, 1>(pl, u, b, coef, vscale, dinv, s);
    case 2 * 16 + 2: return var_pair_impl<2, 2>(pl, u, b, coef, vscale, dinv, s);
    case 2 * 16 + 3: return var_pair_impl<2, 3>(pl, u, b, coef, vscale, dinv, s);
    case 3 * 16 + 1: return var_pair_impl<3, 1>(pl, u, b, coef, vscale, dinv, s);
    case 3 * 16 + 2: return var_pair_impl<3, 2>(pl, u, b, coef, vscale, dinv, s);
    case 3 * 16 + 3: return var_pair_impl<3, 3>(pl, u, b, coef, vscale, dinv, s);
    default: return GMG_ERR_UNSUPPORTED;
  }
}

}  // namespace gmg
