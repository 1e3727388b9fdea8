// Closure form of the patch sweep, two patches per thread (pair_arith.cuh),
// for the arithmetic PA of the including file: whole colours, batches of
// problems, patch lists (slabs, Algorithm 5) and the solve-only mode of
// Algorithm 3, in 2D and 3D.  With one patch per thread the FP32 kernel issued
// two instructions beside each multiply-add; per sweep, before -> now (us):
// FP32 Q4 64^3 934 -> 582, FP64 2D Q3 1024^2 967 -> 693, FP64 closure form Q4
// 64^3 4930 -> 4220.
//
// Patch local_update (Sec. 3.1; Algorithm 4 runs it for every patch of one
// colour per launch):
//   gather    closure bar u_j ((2k+1)^d nodes) into shared memory
//   evaluate  r = h^{2-d} b_j - [A_ref bar u_j]_interior by sum factorisation
//             over the patch: the patch operator is a sum of tensor products
//             of the two-cell 1D matrices M_p, K_p (interior rows x closure
//             columns)
//   solve     d = (T x .. x T) diag(1/sum lambda) (T x .. x T)^T r
//             (fast diagonalisation, App. A.3)
//   scatter   u_interior += omega d  (same-colour interiors are disjoint)
#pragma once
#include <algorithm>
#include <type_traits>

#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "async.cuh"
#include "kernels.h"
#include "pair_lines.cuh"
#include "patch_dispatch.h"
#include "tma_host.h"

namespace gmg {
namespace {

using T = PA::T;
using V = PA::val;
using E = PA::mem;
constexpr bool DF = sizeof(T) == 8;

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Shared memory: per patch IN, its closure of u and its interior
// of b in rows of XU / XB elements of T ([z][y][x]; with the TMA gather a row
// is the box width: C (resp. M + 1) plus the alignment shift, rounded up to
// 16 bytes, and each box starts on 128 bytes); per pair W, entries of E: the
// two fields of the first contraction, in rows of R entries.  Every later
// stage works in place: a thread reads the whole line it writes.
template <int DIM, int K, bool TMA>
struct ClosureSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1;
  static constexpr int A = 16 / (int)sizeof(T);  // elements per 16 bytes
  static constexpr int XU = TMA ? (C + A - 1 + A - 1) / A * A : C;
  static constexpr int XB = TMA ? XU : M;
  static constexpr int R128 = 128 / (int)sizeof(T);
  static constexpr int rnd(int n) { return (n + R128 - 1) / R128 * R128; }
  static constexpr int NCLO = rnd(DIM == 3 ? C * C * XU : C * XU);
  static constexpr int NBIN = rnd(DIM == 3 ? M * M * XB : M * XB);
  static constexpr int NINT = DIM == 3 ? M * M * M : M * M;
  static constexpr int IN = NCLO + NBIN;
  static constexpr int R = DIM == 3 ? C : M;             // row of W (x)
  static constexpr int F = DIM == 3 ? C * M * R : C * R;  // one field: [z][y][x], z in C, y in M (2D: [y][x])
  static constexpr int bytes(int pp) { return pp * 2 * (IN * (int)sizeof(T) + F * (int)sizeof(E)) + 128; }
  // TMA box bytes of the closure of u and of the interior rows of b
  static constexpr int BOX_U = (DIM == 3 ? C * C * XU : C * XU) * (int)sizeof(T);
  static constexpr int BOX_B = (DIM == 3 ? M * M * XB : M * XB) * (int)sizeof(T);
};

// Tensor maps of the u and b vectors of each table entry (TMA gather).
template <int ME>
struct ClosureMaps {
  CUtensorMap u[ME], b[ME];
};
template <>
struct ClosureMaps<0> {};

// One contraction of a line of C closure values: row(i, M x, K x) per interior
// row i, with the line's values loaded by get(closure index) one cell at a
// time (the cells are mirror images).
template <int K, typename G, typename F>
__device__ __forceinline__ void closure_line(G&& get, F&& row) {
  constexpr int M = 2 * K - 1;
  PA::acc cm = PA::zero(), ck = PA::zero();
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    V v[K + 1];
#pragma unroll
    for (int q = 0; q <= K; ++q) v[q] = get(r ? 2 * K - q : q);
#pragma unroll
    for (int p = 1; p < K; ++p) {
      PA::acc m, s;
      pl_cell_row<K, 0, true, 0>(p, v, m);
      pl_cell_row<K, 1, true, 0>(p, v, s);
      row(r ? M - p : p - 1, PA::value(m), PA::value(s));
    }
    pl_centre<K, 0, 0>(r == 0, v, cm);
    pl_centre<K, 1, 0>(r == 0, v, ck);
  }
  row(K - 1, PA::value(cm), PA::value(ck));
}
// the same for two lines: row(i, M p, K p + M q)
template <int K, typename G, typename H, typename F>
__device__ __forceinline__ void closure_line2(G&& getp, H&& getq, F&& row) {
  constexpr int M = 2 * K - 1;
  PA::acc cm = PA::zero(), ck = PA::zero();
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    V v[K + 1], w[K + 1];
#pragma unroll
    for (int q = 0; q <= K; ++q) {
      v[q] = getp(r ? 2 * K - q : q);
      w[q] = getq(r ? 2 * K - q : q);
    }
#pragma unroll
    for (int p = 1; p < K; ++p) {
      PA::acc m, s;
      pl_cell_row<K, 0, true, 0>(p, v, m);
      pl_cell_row<K, 1, true, 0>(p, v, s);
      pl_cell_row<K, 0, false, 0>(p, w, s);
      row(r ? M - p : p - 1, PA::value(m), PA::value(s));
    }
    pl_centre<K, 0, 0>(r == 0, v, cm);
    pl_centre<K, 1, 0>(r == 0, v, ck);
    pl_centre<K, 0, 0>(r == 0, w, ck);
  }
  row(K - 1, PA::value(cm), PA::value(ck));
}
// residual rows: acc[i] (preset) += (K a1 + M a2)_i
template <int K, typename G, typename H>
__device__ __forceinline__ void closure_line_residual(G&& get1, H&& get2, PA::acc (&acc)[2 * K - 1]) {
  constexpr int M = 2 * K - 1;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    V v[K + 1], w[K + 1];
#pragma unroll
    for (int q = 0; q <= K; ++q) {
      v[q] = get1(r ? 2 * K - q : q);
      w[q] = get2(r ? 2 * K - q : q);
    }
#pragma unroll
    for (int p = 1; p < K; ++p) {
      pl_cell_row<K, 1, false, 0>(p, v, acc[r ? M - p : p - 1]);
      pl_cell_row<K, 0, false, 0>(p, w, acc[r ? M - p : p - 1]);
    }
    pl_centre<K, 1, 0>(r == 0, v, acc[K - 1]);
    pl_centre<K, 0, 0>(r == 0, w, acc[K - 1]);
  }
}

// One colour of the sweep.  A CTA takes one group of 2 PP consecutive patches
// of a table entry; a thread carries the same line of patches 2q and 2q + 1.
// Small CTAs, several to an SM, overlap one another's gathers and barriers,
// and the hardware hands them out as SMs become free (persistent CTAs with a
// fixed share: 0.63 against 0.60 ms per FP32 Q4 64^3 sweep, a second input
// buffer 0.66).  The gather is one TMA box per patch and vector (ME > 0:
// tiled cp.async.bulk.tensor loads completing on an mbarrier; the box starts
// at the closure origin rounded down to 16 bytes and the shift is kept per
// patch) or one cp.async per element (ME = 0).  The last contraction runs along the slowest
// axis, as does the scatter: consecutive lanes then hold consecutive x, and
// loads and stores touch whole sectors.  Stages, 3D (2D: without z; y takes
// the part of z):
//   y: P,Q (on -u) | x: A1,A2 | z: r = h^{2-d} b + K_z A1 + M_z A2, forward z
//   y: forward | x: forward, diagonal, backward | y: backward
//   z: backward, u_new = u_old + omega d
// FP64 3D: the local solver is exact, so the updated interior A_j^{-1} (b_j -
// bar A_j bar u_j) + u_j equals A_j^{-1} (b_j - bar A_j bar u_j^0), bar u_j^0
// the closure with its interior set to zero: the residual is evaluated with a
// zero interior and the scatter writes omega d + (1 - omega) u_j.  (FP32 keeps
// the correction form: recomputing the interior would cost a factor
// cond(A_j) in single precision.)
// Same-colour patches never write each other's closure, so the buffered
// closure values are the values the gather (eq. "gather") reads.
template <int DIM, int K, int NT, int PP, int CTAS, int ME>
__global__ void __launch_bounds__(NT, CTAS) pair_closure_kernel(const __grid_constant__ PatchTable tab,
                                                                const T* __restrict__ dinv,
                                                                const __grid_constant__ ClosureMaps<ME> maps,
                                                                int* __restrict__ err) {
  constexpr bool TMA = ME > 0;
  constexpr bool EXACT = DF && DIM == 3;
  using Z = ClosureSmem<DIM, K, TMA>;
  constexpr int C = Z::C, M = Z::M, XU = Z::XU, XB = Z::XB, R = Z::R, F = Z::F, NP = 2 * PP;
  constexpr int LINES = DIM == 3 ? M * M : M;  // interior lines per axis
  static_assert(NP <= NT, "one lane issues the copies of one patch");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  T* const IN = reinterpret_cast<T*>(smem_raw + ((128 - (async::smem_u32(smem_raw) & 127)) & 127));  // [NP][IN]
  E* const W = reinterpret_cast<E*>(IN + NP * Z::IN);  // [PP][2][F]
  __shared__ long long s_origin[NP];
  __shared__ int s_shift[NP];  // of the closure inside its TMA box
  __shared__ __align__(8) uint64_t s_bar;
  const int mode = tab.mode, grp = blockIdx.x;
  // element offsets inside a patch's input: closure of u, interior of b
  auto uo = [](int x, int y, int z) { return DIM == 3 ? (z * C + y) * XU + x : y * XU + x; };
  auto bo = [](int x, int y, int z) { return DIM == 3 ? (z * M + y) * XB + x : y * XB + x; };

  int entry = 0, hi = tab.n - 1;  // last table entry with group_begin <= grp
  while (entry < hi) {
    const int mid = (entry + hi + 1) >> 1;
    if (tab.e[mid].group_begin <= grp) entry = mid;
    else hi = mid - 1;
  }
  const PatchEntry& e = tab.e[entry];
  const int g = grp - e.group_begin, nv = min(NP, e.n_patches - g * NP), npair = (nv + 1) / 2;
  T* __restrict__ const u = static_cast<T*>(e.u);
  const long long py = e.py, pz = e.pz;
  const float sb = (float)e.sb;  // h^{2-d}: n in 3D, 1 in 2D, exact in float
  if (TMA) {
    if (threadIdx.x == 0) {
      async::mbar_init(&s_bar, 1);
      async::mbar_arrive_expect_tx(&s_bar, (uint32_t)(nv * ((mode == 0 ? Z::BOX_U : 0) + Z::BOX_B)));
    }
    __syncthreads();
  }
  {
    // patch origins and copies: the patches are spread over the warps, as a
    // warp issues its lanes' copies one after the other
    const int q = threadIdx.x / 32 + (threadIdx.x % 32) * (NT / 32);
    if (q < nv) {
      int pid = g * NP + q;
      if (e.plist) pid = e.plist[pid];
      const int i0 = pid % e.count[0], rest = pid / e.count[0];
      const int i1 = rest % e.count[1], i2 = DIM == 3 ? rest / e.count[1] : 0;
      const int o0 = (e.first[0] + 2 * i0 - 1) * K, o1 = (e.first[1] + 2 * i1 - 1) * K;
      const int o2 = DIM == 3 ? (e.first[2] + 2 * i2 - 1) * K : 0;
      s_origin[q] = o0 + py * o1 + pz * o2;
      s_shift[q] = TMA ? o0 % Z::A : 0;
      if constexpr (TMA) {
        T* const dst = IN + q * Z::IN;
        const int xa = o0 - o0 % Z::A;
        if (DIM == 3) {
          if (mode == 0) async::tma_load_3d(dst, &maps.u[entry], xa, o1, o2, &s_bar);
          async::tma_load_3d(dst + Z::NCLO, &maps.b[entry], xa, o1 + 1, o2 + 1, &s_bar);
        } else {
          if (mode == 0) async::tma_load_2d(dst, &maps.u[entry], xa, o1, &s_bar);
          async::tma_load_2d(dst + Z::NCLO, &maps.b[entry], xa, o1 + 1, &s_bar);
        }
      }
    }
  }
  __syncthreads();
  bool wait_ok = true;  // an expired wait is recorded and the kernel carries on
  if constexpr (TMA) {
    wait_ok = async::mbar_wait(&s_bar, 0);
  } else {
    const T* __restrict__ b = static_cast<const T*>(e.b);
    constexpr int NC = DIM == 3 ? C * C * C : C * C;
    auto copy = [](T* d, const T* s) {
      asm volatile("cp.async.ca.shared.global [%0], [%1], %2;\n" ::"r"(async::smem_u32(d)), "l"(s), "n"(sizeof(T)) : "memory");
    };
    // the solve-only mode needs no closure: only the residual's interior
    for (int t = threadIdx.x; t < (mode == 0 ? nv * NC : 0); t += NT) {
      const int p = t / NC, l = t % NC, x = l % C, row = l / C;
      copy(IN + p * Z::IN + l, u + s_origin[p] + x + py * (row % C) + (DIM == 3 ? pz * (row / C) : 0));
    }
    for (int t = threadIdx.x; t < nv * Z::NINT; t += NT) {
      const int p = t / Z::NINT, l = t % Z::NINT, x = l % M, row = l / M;
      copy(IN + p * Z::IN + Z::NCLO + l, b + s_origin[p] + 1 + x + py * (row % M + 1) + (DIM == 3 ? pz * (row / M + 1) : 0));
    }
    async::copy_wait_all();
    __syncthreads();
  }
  // both patches' inputs, shifted to the closure origin (a lone last patch
  // has whatever the buffer holds beside it; nothing of that is stored)
  auto input = [&](int q, int second) -> const T* {
    const int p = 2 * q + second;
    return IN + p * Z::IN + (p < nv ? s_shift[p] : 0);
  };

  if (mode == 0) {
    if (DIM == 3) {
      // ---- y: P = M_y u, Q = K_y u on lines (x, z), from -u ----
      constexpr int CI = C - 2;
      for (int t = threadIdx.x; t < npair * C * C; t += NT) {
        int q, x, z;
        bool inner = false;
        if (EXACT) {
          // interior lines first, pairs interleaved: a warp runs one kind of
          // line (with a zero interior an inner line has only its end values)
          q = t % npair;
          const int lp = t / npair;
          inner = lp < CI * CI;
          if (inner) {
            x = 1 + lp % CI;
            z = 1 + lp / CI;
          } else {
            const int o = lp - CI * CI;
            if (o < C) { x = o; z = 0; }
            else if (o < 2 * C) { x = o - C; z = C - 1; }
            else { x = ((o - 2 * C) & 1) ? C - 1 : 0; z = 1 + (o - 2 * C) / 2; }
          }
        } else {
          q = t / (C * C);
          x = t % (C * C) % C;
          z = t % (C * C) / C;
        }
        const T* const a = input(q, 0) + uo(x, 0, z);
        const T* const b = input(q, 1) + uo(x, 0, z);
        E* const P = W + q * 2 * F + z * M * R + x;
        auto get = [&](int y) -> V { return PA::pack_neg(a[y * XU], b[y * XU]); };
        auto put = [&](int j, V m, V k) {
          PA::store(P[j * R], m);
          PA::store(P[F + j * R], k);
        };
        if (EXACT && inner) {
          const V u0 = get(0), uc = get(C - 1);
#pragma unroll
          for (int j = 0; j < M; ++j) {
            const int o = pl_off_patch(K) + j * C;
            PA::acc m, k;
            if (j <= K - 1) {
              m = PA::first(pl_coef(p_M[o]), u0);
              k = PA::first(pl_coef(p_K[o]), u0);
            }
            if (j == K - 1) {
              PA::add(m, pl_coef(p_M[o + C - 1]), uc);
              PA::add(k, pl_coef(p_K[o + C - 1]), uc);
            } else if (j > K - 1) {
              m = PA::first(pl_coef(p_M[o + C - 1]), uc);
              k = PA::first(pl_coef(p_K[o + C - 1]), uc);
            }
            put(j, PA::value(m), PA::value(k));
          }
        } else {
          closure_line<K>(get, put);
        }
      }
      __syncthreads();
      // ---- x: A1 = M_x P, A2 = K_x P + M_x Q on rows (y, z), in place ----
      for (int t = threadIdx.x; t < npair * C * M; t += NT) {
        E* const P = W + t / (C * M) * 2 * F + t % (C * M) * R;
        V a1[M], a2[M];
        closure_line2<K>([&](int x) -> V { return PA::load(P[x]); }, [&](int x) -> V { return PA::load(P[F + x]); },
                         [&](int i, V m, V k) {
                           a1[i] = m;
                           a2[i] = k;
                         });
#pragma unroll
        for (int i = 0; i < M; ++i) {
          PA::store(P[i], a1[i]);
          PA::store(P[F + i], a2[i]);
        }
      }
    } else {
      // ---- x: P = M_x u, Q = K_x u on rows y, from -u ----
      for (int t = threadIdx.x; t < npair * C; t += NT) {
        const int q = t / C, y = t % C;
        const T* const a = input(q, 0) + uo(0, y, 0);
        const T* const b = input(q, 1) + uo(0, y, 0);
        E* const P = W + q * 2 * F + y * R;
        closure_line<K>([&](int x) -> V { return PA::pack_neg(a[x], b[x]); },
                        [&](int i, V m, V k) {
                          PA::store(P[i], m);
                          PA::store(P[F + i], k);
                        });
      }
    }
    __syncthreads();
  }

  // ---- residual on interior lines of the slowest axis (z in 3D, y in 2D),
  // then the forward transform along it, in place of the first field ----
  constexpr int SL = DIM == 3 ? M * R : R;  // stride of the line in W
  auto line = [&](int q, int ln) -> E* { return W + q * 2 * F + (DIM == 3 ? ln / M * R + ln % M : ln); };
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;  // 3D: x + M y; 2D: x
    const int bofs = Z::NCLO + (TMA ? 1 : 0) + (DIM == 3 ? bo(ln % M, ln / M, 0) : ln);
    const T* const ba = input(q, 0) + bofs;
    const T* const bb = input(q, 1) + bofs;
    PA::acc acc[M];
#pragma unroll
    for (int l = 0; l < M; ++l) {
      const int o = (DIM == 3 ? M * XB : XB) * l;
      acc[l] = PA::scaled(sb, PA::pack(ba[o], bb[o]));
    }
    if (mode == 0) {
      const E* const A = line(q, ln);
      closure_line_residual<K>([&](int s) -> V { return PA::load(A[s * SL]); },
                               [&](int s) -> V { return PA::load(A[F + s * SL]); }, acc);
    }
    V r[M];
#pragma unroll
    for (int l = 0; l < M; ++l) r[l] = PA::value(acc[l]);
    E* const w = line(q, ln);
    pl_forward<K>(r, [&](int l, V v) { PA::store(w[l * SL], v); });
  }
  __syncthreads();
  // ---- local solve by fast diagonalisation (App. A.3), in place ----
  auto line_y = [&](auto forward) {
    for (int t = threadIdx.x; t < npair * LINES; t += NT) {
      const int q = t / LINES, ln = t % LINES;
      E* const w = W + q * 2 * F + ln % M + ln / M * M * R;
      V v[M];
#pragma unroll
      for (int j = 0; j < M; ++j) v[j] = PA::load(w[j * R]);
      auto put = [&](int j, V x) { PA::store(w[j * R], x); };
      if constexpr (decltype(forward)::value) pl_forward<K>(v, put);
      else pl_backward<K>(v, put);
    }
    __syncthreads();
  };
  if (DIM == 3) line_y(std::true_type());
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;  // 3D: y + M z; 2D: y
    E* const w = W + q * 2 * F + ln * R;
    V v[M];
#pragma unroll
    for (int i = 0; i < M; ++i) v[i] = PA::load(w[i]);
    // the diagonal is symmetric in its indices: entry (.., i), so that
    // consecutive lanes read consecutive values
    V x[M];
    pl_forward<K>(v, [&](int i, V y) { x[i] = PA::diagonal(dinv, Z::NINT, i * LINES + ln, y); });
    pl_backward<K>(x, [&](int i, V y) { PA::store(w[i], y); });
  }
  __syncthreads();
  if (DIM == 3) line_y(std::false_type());
  // ---- backward along the slowest axis and scatter (eq. "scatter") ----
  const T om = (T)tab.omega;
  const long long ps = DIM == 3 ? pz : py;
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;
    const E* const w = line(q, ln);
    V v[M];
#pragma unroll
    for (int l = 0; l < M; ++l) v[l] = PA::load(w[l * SL]);
    const bool two = 2 * q + 1 < nv;
    const int x = 1 + ln % M, y = DIM == 3 ? 1 + ln / M : 0;
    const long long ofs = x + (DIM == 3 ? py * y : 0) + ps;
    const int uofs = DIM == 3 ? uo(x, y, 1) : uo(x, 1, 0);
    constexpr int US = DIM == 3 ? C * XU : XU;  // the slow stride of the closure
    T* const ga = u + s_origin[2 * q] + ofs;
    T* const gb = two ? u + s_origin[2 * q + 1] + ofs : ga;
    const T *const ia = input(q, 0) + uofs, *const ib = input(q, 1) + uofs;
    pl_backward<K>(v, [&](int l, V d) {
      auto one = [&](T* g, const T* i, T dv) {
        *g = EXACT && mode == 0 ? fma(om, dv, (T(1) - om) * *i) : fma(om, dv, mode == 0 ? *i : *g);
      };
      one(ga + ps * l, ia + US * l, PA::x(d));
      if (two) one(gb + ps * l, ib + US * l, PA::y(d));
    });
  }
  if (!wait_ok) atomicExch(err, GMG_ERR_TIMEOUT);
}

// ---- host side ----

// Patch pairs and threads per CTA, and the CTAs per SM that the registers are
// limited for.  A pair has LINES lines in most stages, and a CTA as many pairs
// as fill its threads with them.  Measured per sweep (us), the shape taken
// first: FP32 Q3 64^3 1 pair in 32 threads 279, 2 in 64 296, 5 in 128 361; Q4
// 64^3 1 in 64 582, 2 in 128 630, 4 in 224 787; Q6 40^3 with registers for 3
// CTAs 594, without 770; FP64 Q3 64^3 5 in 128 1536, 1 in 32 1826; FP64 2D Q3
// 1024^2 25 in 128 697, 12 in 64 756; FP32 2D Q3 6 in 32 201, 25 in 128 238.
template <int DIM, int K>
struct ClosureCfg {
  static constexpr int M = 2 * K - 1, LINES = DIM == 3 ? M * M : M;
  static constexpr int NT = DIM == 2 ? (!DF ? 32 : K == 2 ? 64 : 128)
                          : K <= 3 ? (DF ? 128 : 32) : K >= 7 ? 256 : (LINES + 31) / 32 * 32;
  static constexpr int PP = cmax(1, std::min(NT / LINES, 3 * NT / 8));
  static constexpr int CTAS = DIM == 2 ? (DF && K == 3 ? 4 : 1) : !DF && K == 5 ? 6 : !DF && K == 6 ? 3 : 1;
};
// a pair of the largest FP64 patches does not fit in the shared memory of a CTA
template <int DIM, int K>
constexpr bool closure_pairs() {
  return ClosureSmem<DIM, K, true>::bytes(1) <= 227 * 1024;
}

template <int DIM, int K, int PP, int NT, int CTAS, int ME>
int closure_launch(PatchTable& tab, const T* dinv, cudaStream_t s) {
  using Z = ClosureSmem<DIM, K, (ME > 0)>;
  constexpr int SMEM = Z::bytes(PP);
  static_assert(SMEM <= 227 * 1024, "sweep kernel shared memory exceeds the per-CTA limit");
  auto kern = pair_closure_kernel<DIM, K, NT, PP, CTAS, ME>;
  static PerDevice<bool> ready_dev;  // attribute set once per device
  bool* const ready = ready_dev.get();
  if (!ready) return GMG_ERR_CUDA;
  if (!*ready) {
    if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess)
      return GMG_ERR_CUDA;
    *ready = true;
  }
  int groups = 0;
  for (int i = 0; i < tab.n; ++i) {
    tab.e[i].group_begin = groups;
    groups += (tab.e[i].n_patches + 2 * PP - 1) / (2 * PP);
  }
  tab.total_groups = groups;
  if (groups <= 0) return GMG_OK;
  ClosureMaps<ME> maps;
  if constexpr (ME > 0) {
    for (int i = 0; i < tab.n; ++i) {
      const PatchEntry& e = tab.e[i];
      if (!tma_encode(&maps.u[i], e.u, (int)sizeof(T), DIM, e.N, e.py, e.pz, Z::XU, Z::C) ||
          !tma_encode(&maps.b[i], e.b, (int)sizeof(T), DIM, e.N, e.py, e.pz, Z::XB, Z::M))
        return GMG_ERR_CUDA;
    }
  }
  int* const flag = device_wait_flag();
  if (!flag) return GMG_ERR_CUDA;
  kern<<<groups, NT, SMEM, s>>>(tab, dinv, maps, flag);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

// the TMA gather when every vector of the table allows the boxes, else one
// cp.async per element
template <int DIM, int K, int PP, int NT, int CTAS>
int closure_gather(PatchTable& tab, const T* dinv, cudaStream_t s) {
  bool tma = true;
  for (int i = 0; i < tab.n; ++i) {
    const PatchEntry& e = tab.e[i];
    if (e.N < 2 || !tma_vector_ok(e.u, (int)sizeof(T), DIM, e.py, e.pz) ||
        !tma_vector_ok(e.b, (int)sizeof(T), DIM, e.py, e.pz))
      tma = false;
  }
  if (!tma) return closure_launch<DIM, K, PP, NT, CTAS, 0>(tab, dinv, s);
  if (tab.n == 1) return closure_launch<DIM, K, PP, NT, CTAS, 1>(tab, dinv, s);
  return closure_launch<DIM, K, PP, NT, CTAS, kMaxTable>(tab, dinv, s);
}

template <int DIM, int K>
int closure_table(PatchTable& tab, const T* dinv, int ppc, cudaStream_t s) {
  using Cfg = ClosureCfg<DIM, K>;
  // tuned patches-per-CTA variants of the batched sweep (patches come in pairs)
  if constexpr (DIM == 3 && !DF && K <= 4) {
    if (ppc == 1) return closure_gather<DIM, K, 1, 32, 1>(tab, dinv, s);
    if (ppc == 2) return closure_gather<DIM, K, 1, 64, 1>(tab, dinv, s);
    if (ppc == 4) return closure_gather<DIM, K, 2, 128, 1>(tab, dinv, s);
  }
  return closure_gather<DIM, K, Cfg::PP, Cfg::NT, Cfg::CTAS>(tab, dinv, s);
}

}  // namespace
}  // namespace gmg
