// Variable-coefficient patch sweep (degree <= 3), two patches per thread
// (pair_arith.cuh), for the arithmetic PA of the including file; patches
// without a learned correction (those with one take patch_var_kernel).
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

#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "async.cuh"
#include "kernels.h"
#include "pair_lines.cuh"
#include "tma_host.h"

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

// Shared memory per patch: closure of u, interior of b (TMA boxes, or rows of
// C and M elements without TMA); per pair the two fields of a contraction,
// [z][y][x] with 2k rows per contracted axis; stages work in place.
template <int DIM, int K, bool TMA>
struct VarSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1, H = 2 * K;
  static constexpr int A = 16 / (int)sizeof(T);
  static constexpr int XU = TMA ? (C + A - 1 + A - 1) / A * A : C;
  static constexpr int XB = TMA ? XU : M;
  static constexpr int R128 = 128 / (int)sizeof(T);
  static constexpr int rnd(int n) { return (n + R128 - 1) / R128 * R128; }
  static constexpr int NCLO = rnd(DIM == 3 ? C * C * XU : C * XU);
  static constexpr int NBIN = rnd(DIM == 3 ? M * M * XB : M * XB);
  static constexpr int NINT = DIM == 3 ? M * M * M : M * M;
  static constexpr int IN = NCLO + NBIN;
  static constexpr int R = DIM == 3 ? C : H;             // row (x)
  static constexpr int F = DIM == 3 ? C * H * R : C * R;  // one field
  static constexpr int NCELL = 1 << DIM;
  static constexpr int bytes(int pp) {
    return pp * (2 * IN * (int)sizeof(T) + (2 * F + NCELL) * (int)sizeof(E)) + 128;
  }
  static constexpr int BOX_U = (DIM == 3 ? C * C * XU : C * XU) * (int)sizeof(T);
  static constexpr int BOX_B = (DIM == 3 ? M * M * XB : M * XB) * (int)sizeof(T);
};

struct VarArgs {
  PatchLaunch pl;
  T* u;
  const T* b;
  const T* coef;
  const T* vscale;  // abar, theta per interior vertex
  const T* dinv;
  int* err;
};
struct VarMaps {
  CUtensorMap u, b;
};

// A CTA takes 2 PP consecutive patches of the colour, a thread the same line
// of patches 2q and 2q + 1.  Stages, 3D (2D: without the first, and y for z):
//   y: P, Q (on -u), 2k rows | x: A1, A2, 2k rows each way |
//   z: a_c (K_z A1 + M_z A2) per column of a cell pair |
//   z: r = h^{2-d} b + the columns of a node (1, 2 or 4), forward transform |
//   y: forward | x: forward, diagonal, backward | y: backward |
//   z: backward, u += omega theta / abar d
template <int DIM, int K, int NT, int PP, bool TMA>
__global__ void __launch_bounds__(NT) pair_var_kernel(const __grid_constant__ VarArgs va,
                                                      const __grid_constant__ VarMaps maps) {
  using Z = VarSmem<DIM, K, TMA>;
  constexpr int C = Z::C, M = Z::M, H = Z::H, XU = Z::XU, XB = Z::XB, R = Z::R, F = Z::F, NP = 2 * PP;
  constexpr int LINES = DIM == 3 ? M * M : M, NCELL = Z::NCELL;
  static_assert(NP <= NT, "one lane issues the copies of one patch");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* const IN = reinterpret_cast<T*>(smem_raw + ((128 - (async::smem_u32(smem_raw) & 127)) & 127));  // [NP][IN]
  E* const W = reinterpret_cast<E*>(IN + NP * Z::IN);  // [PP][2][F]
  E* const CO = W + PP * 2 * F;                         // [PP][NCELL] cell coefficients of both patches
  __shared__ long long s_origin[NP];
  __shared__ int s_shift[NP], s_vert[NP][3];
  __shared__ T s_scale[NP];
  __shared__ __align__(8) uint64_t s_bar;
  const PatchLaunch& pl = va.pl;
  const long long py = pl.g.py, pz = pl.g.pz;
  const int g0 = blockIdx.x * NP, nv = min(NP, pl.n_patches - g0), npair = (nv + 1) / 2, n = pl.g.n;
  const float sb = (float)pl.sb;  // an integer power of the cell count, exact in float
  auto uo = [](int x, int y, int z) { return DIM == 3 ? (z * C + y) * XU + x : y * XU + x; };
  auto bo = [](int x, int y, int z) { return DIM == 3 ? (z * M + y) * XB + x : y * XB + x; };
  if (TMA) {
    if (threadIdx.x == 0) {
      async::mbar_init(&s_bar, 1);
      async::mbar_arrive_expect_tx(&s_bar, (uint32_t)(nv * (Z::BOX_U + Z::BOX_B)));
    }
    __syncthreads();
  }
  {
    const int q = threadIdx.x / 32 + (threadIdx.x % 32) * (NT / 32);  // the patches are spread over the warps
    if (q < nv) {
      const int pid = g0 + q;
      const int i0 = pid % pl.count[0], rest = pid / pl.count[0];
      const int i1 = rest % pl.count[1], i2 = DIM == 3 ? rest / pl.count[1] : 0;
      const int v0 = pl.first[0] + 2 * i0, v1 = pl.first[1] + 2 * i1, v2 = DIM == 3 ? pl.first[2] + 2 * i2 : 1;
      const int o0 = (v0 - 1) * K, o1 = (v1 - 1) * K, o2 = (v2 - 1) * K;
      s_origin[q] = o0 + py * o1 + (DIM == 3 ? pz * o2 : 0);
      s_shift[q] = TMA ? o0 % Z::A : 0;
      s_vert[q][0] = v0 - 1;
      s_vert[q][1] = v1 - 1;
      s_vert[q][2] = v2 - 1;
      if constexpr (TMA) {
        T* const dst = IN + q * Z::IN;
        const int xa = o0 - o0 % Z::A;
        if (DIM == 3) {
          async::tma_load_3d(dst, &maps.u, xa, o1, o2, &s_bar);
          async::tma_load_3d(dst + Z::NCLO, &maps.b, xa, o1 + 1, o2 + 1, &s_bar);
        } else {
          async::tma_load_2d(dst, &maps.u, xa, o1, &s_bar);
          async::tma_load_2d(dst + Z::NCLO, &maps.b, xa, o1 + 1, &s_bar);
        }
      }
      const long long vid = (v0 - 1) + (long long)(n - 1) * ((v1 - 1) + (DIM == 3 ? (long long)(n - 1) * (v2 - 1) : 0));
      s_scale[q] = (T)pl.omega * va.vscale[2 * vid + 1] / va.vscale[2 * vid];
    }
  }
  __syncthreads();
  for (int t = threadIdx.x; t < npair * NCELL; t += NT) {
    const int q = t / NCELL, c = t % NCELL;
    auto cell = [&](int p) -> T {
      return va.coef[s_vert[p][0] + (c & 1) + (long long)n * ((s_vert[p][1] + ((c >> 1) & 1)) +
                                                             (DIM == 3 ? (long long)n * (s_vert[p][2] + (c >> 2)) : 0))];
    };
    PA::store(CO[t], PA::pack(cell(2 * q), cell(2 * q + 1 < nv ? 2 * q + 1 : 2 * q)));
  }
  bool wait_ok = true;  // an expired wait is recorded and the kernel carries on
  if constexpr (TMA) {
    wait_ok = async::mbar_wait(&s_bar, 0);
  } else {  // element by element
    constexpr int NC = DIM == 3 ? C * C * C : C * C;
    for (int t = threadIdx.x; t < nv * NC; t += NT) {
      const int p = t / NC, l = t % NC, x = l % C, row = l / C;
      IN[p * Z::IN + l] = va.u[s_origin[p] + x + py * (row % C) + (DIM == 3 ? pz * (row / C) : 0)];
    }
    for (int t = threadIdx.x; t < nv * Z::NINT; t += NT) {
      const int p = t / Z::NINT, l = t % Z::NINT, x = l % M, row = l / M;
      IN[p * Z::IN + Z::NCLO + l] =
          va.b[s_origin[p] + 1 + x + py * (row % M + 1) + (DIM == 3 ? pz * (row / M + 1) : 0)];
    }
  }
  __syncthreads();  // (also the coefficients)
  // (a lone last patch has whatever the buffer holds beside it; nothing of
  // that is stored)
  auto input = [&](int q, int second) -> const T* {
    const int p = 2 * q + second;
    return IN + p * Z::IN + (p < nv ? s_shift[p] : 0);
  };
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
      const T *const a = input(q, 0) + uo(x, 0, z), *const b = input(q, 1) + uo(x, 0, z);
      E* const P = W + q * 2 * F + z * H * R + x;
      line_rows([&](int y) -> V { return PA::pack_neg(a[y * XU], b[y * XU]); },
                [&](int j, V m, V k) {
                  PA::store(P[j * R], m);
                  PA::store(P[F + j * R], k);
                });
    }
    __syncthreads();
    // ---- x: A1 = M_x P, A2 = K_x P + M_x Q on rows (y, z), in place ----
    for (int t = threadIdx.x; t < npair * C * H; t += NT) {
      E* const P = W + t / (C * H) * 2 * F + t % (C * H) * R;
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
      const T *const a = input(q, 0) + uo(0, y, 0), *const b = input(q, 1) + uo(0, y, 0);
      E* const P = W + q * 2 * F + y * R;
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
    E* const P = W + q * 2 * F + (DIM == 3 ? Y * R : 0) + X;
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
    return W + q * 2 * F + (DIM == 3 ? pos(ln / M) * R + pos(ln % M) : pos(ln));
  };
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES, i = ln % M, j = ln / M;
    const int bofs = Z::NCLO + (TMA ? 1 : 0) + (DIM == 3 ? bo(i, j, 0) : i);
    const T *const ba = input(q, 0) + bofs, *const bb = input(q, 1) + bofs;
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
      const int o = (DIM == 3 ? M * XB : XB) * l;
      r[l] = PA::sum(PA::value(PA::scaled(sb, PA::pack(ba[o], bb[o]))), s);
    }
    pl_forward<K>(r, [&](int l, V v) { PA::store(w[l * SL], v); });
  }
  __syncthreads();
  // ---- local solve by fast diagonalisation (App. A.3), in place ----
  auto line_y = [&](auto forward) {
    for (int t = threadIdx.x; t < npair * LINES; t += NT) {
      const int q = t / LINES, ln = t % LINES;  // x + M z
      E* const w = W + q * 2 * F + ln / M * SL + pos(ln % M);
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
    E* const w = W + q * 2 * F + (DIM == 3 ? ln / M * SL + pos(ln % M) * R : ln * SL);
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
  const long long ps = DIM == 3 ? pz : py;
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;
    const E* const w = column(q, ln);
    V v[M];
#pragma unroll
    for (int l = 0; l < M; ++l) v[l] = PA::load(w[l * SL]);
    const bool two = 2 * q + 1 < nv;
    const int x = 1 + ln % M, y = DIM == 3 ? 1 + ln / M : 0;
    const long long ofs = x + (DIM == 3 ? py * y : 0) + ps;
    const int uofs = DIM == 3 ? uo(x, y, 1) : uo(x, 1, 0);
    constexpr int US = DIM == 3 ? C * XU : XU;
    T* const ga = va.u + s_origin[2 * q] + ofs;
    T* const gb = two ? va.u + s_origin[2 * q + 1] + ofs : ga;
    const T *const ia = input(q, 0) + uofs, *const ib = input(q, 1) + uofs;
    const T sa = s_scale[2 * q], sc = two ? s_scale[2 * q + 1] : T(0);
    pl_backward<K>(v, [&](int l, V d) {
      ga[ps * l] = fma(sa, PA::x(d), ia[US * l]);
      if (two) gb[ps * l] = fma(sc, PA::y(d), ib[US * l]);
    });
  }
  if (!wait_ok) atomicExch(va.err, GMG_ERR_TIMEOUT);
}

// ---- host side ----

// patch pairs and threads per CTA: as many pairs as fill the threads with the
// interior lines of a stage
template <int DIM, int K>
struct VarPairCfg {
  static constexpr int LINES = DIM == 3 ? (2 * K - 1) * (2 * K - 1) : 2 * K - 1;
#ifdef VPP
  static constexpr int NT = VNT, PP = VPP;
#else
  static constexpr int NT = DF || DIM == 2 ? 128 : 32;
  static constexpr int PP = std::max(1, std::min(NT / LINES, 3 * NT / 8));
#endif
};

template <int DIM, int K, bool TMA>
int var_launch(const VarArgs& va, const VarMaps& maps, cudaStream_t s) {
  using Cfg = VarPairCfg<DIM, K>;
  constexpr int SMEM = VarSmem<DIM, K, TMA>::bytes(Cfg::PP);
  static_assert(SMEM <= 227 * 1024, "sweep kernel shared memory exceeds the per-CTA limit");
  auto kern = pair_var_kernel<DIM, K, Cfg::NT, Cfg::PP, TMA>;
  static PerDevice<bool> ready_dev;  // attribute set once per device
  bool* const ready = ready_dev.get();
  if (!ready) return GMG_ERR_CUDA;
  if (!*ready) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess)
      return GMG_ERR_CUDA;
    *ready = true;
  }
  kern<<<(va.pl.n_patches + 2 * Cfg::PP - 1) / (2 * Cfg::PP), Cfg::NT, SMEM, s>>>(va, maps);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

template <int DIM, int K>
int var_pair_impl(const PatchLaunch& pl, T* u, const T* b, const T* coef, const T* vscale, const T* dinv,
                  cudaStream_t s) {
  if (pl.n_patches <= 0) return GMG_OK;
  VarArgs va{pl, u, b, coef, vscale, dinv, device_wait_flag()};
  if (!va.err) return GMG_ERR_CUDA;
  VarMaps maps{};
  constexpr int es = (int)sizeof(T);
  if (!tma_vector_ok(u, es, DIM, pl.g.py, pl.g.pz) || !tma_vector_ok(b, es, DIM, pl.g.py, pl.g.pz))
    return var_launch<DIM, K, false>(va, maps, s);
  using Z = VarSmem<DIM, K, true>;
  if (!tma_encode(&maps.u, u, es, DIM, pl.g.N, pl.g.py, pl.g.pz, Z::XU, Z::C) ||
      !tma_encode(&maps.b, b, es, DIM, pl.g.N, pl.g.py, pl.g.pz, Z::XB, Z::M))
    return GMG_ERR_CUDA;
  return var_launch<DIM, K, true>(va, maps, s);
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
