// Closure form of the patch sweep, PA::W patches per thread (pair_arith.cuh: two,
// or one where that is faster, see SoloCfg), for the arithmetic PA of the
// including file: whole colours, batches of problems, patch lists (slabs,
// Algorithm 5) and the solve-only mode of Algorithm 3, in 2D and 3D.  With one patch per thread the FP32 kernel issued
// two instructions beside each multiply-add; per sweep, before -> now (us):
// FP32 Q4 64^3 934 -> 583, FP64 closure form Q4 64^3 4930 -> 3180.
//
// Patch local_update (Sec. 3.1; Algorithm 4 runs it for every patch of one
// colour per launch):
//   gather    closure bar u_j ((2k+1)^d nodes)
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

#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "kernels.h"
#include "pair_lines.cuh"
#include "patch_dispatch.h"

namespace gmg {
namespace {

using T = PA::T;
using V = PA::val;
using E = PA::mem;
constexpr bool DF = sizeof(T) == 8;

__host__ __device__ constexpr int cmax(int a, int b) { return a > b ? a : b; }

// Shared memory per pair (one patch with W = 1), entries of E: the two fields of the first
// contraction, in rows of R entries.  Every later stage works in place: a
// thread reads the whole line it writes.  u and b go from global memory
// straight to registers (lanes along x): without room for the closures more
// than twice as many CTAs fit on an SM, which overlap one another's loads and
// barriers (FP32 Q4 64^3: 9 KB a pair against 22 KB with TMA boxes).
template <int DIM, int K>
struct ClosureSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1;
  static constexpr int NINT = DIM == 3 ? M * M * M : M * M;
  static constexpr int R = DIM == 3 ? C : M;             // row of W (x)
  static constexpr int F = DIM == 3 ? C * M * R : C * R;  // one field: [z][y][x], z in C, y in M (2D: [y][x])
  static constexpr int bytes(int pp) { return pp * 2 * F * (int)sizeof(E); }
};

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

// One colour of the sweep.  A CTA takes one group of W PP consecutive patches
// of a table entry; a thread carries the same line of patches 2q and 2q + 1
// (W = 2; the text below says pair for what a thread carries).
// Small CTAs, several to an SM, overlap one another's loads and barriers, and
// the hardware hands them out as SMs become free (persistent CTAs with a fixed
// share: 0.63 against 0.60 ms per FP32 Q4 64^3 sweep).  The last contraction runs along the slowest
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
// Same-colour patches never write each other's closure, so the order in which
// they run does not matter.
template <int DIM, int K, int NT, int PP, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) pair_closure_kernel(const __grid_constant__ PatchTable tab,
                                                                const T* __restrict__ dinv) {
  constexpr bool EXACT = DF && DIM == 3;
  using Z = ClosureSmem<DIM, K>;
  constexpr int C = Z::C, M = Z::M, R = Z::R, F = Z::F, W = PA::W, NP = W * PP;
  constexpr int LINES = DIM == 3 ? M * M : M;  // interior lines per axis
  static_assert(NP <= NT, "one thread sets up one patch");
  extern __shared__ __align__(128) unsigned char smem_raw[];
  E* const S = reinterpret_cast<E*>(smem_raw);  // [PP][2][F]
  __shared__ long long s_origin[NP];
  const int mode = tab.mode, grp = blockIdx.x;
  int entry = 0, hi = tab.n - 1;  // last table entry with group_begin <= grp
  while (entry < hi) {
    const int mid = (entry + hi + 1) >> 1;
    if (tab.e[mid].group_begin <= grp) entry = mid;
    else hi = mid - 1;
  }
  const PatchEntry& e = tab.e[entry];
  const int g = grp - e.group_begin, nv = min(NP, e.n_patches - g * NP), npair = (nv + W - 1) / W;
  T* const u = static_cast<T*>(e.u);
  const T* __restrict__ const b = static_cast<const T*>(e.b);
  const long long py = e.py, pz = e.pz, ps = DIM == 3 ? pz : py;  // ps: the slowest axis
  const float sb = (float)e.sb;  // h^{2-d}: n in 3D, 1 in 2D, exact in float
  if ((int)threadIdx.x < NP) {  // (a lone last patch is carried twice and stored once)
    int pid = g * NP + min((int)threadIdx.x, nv - 1);
    if (e.plist) pid = e.plist[pid];
    const int i0 = pid % e.count[0], rest = pid / e.count[0];
    const int i1 = rest % e.count[1], i2 = DIM == 3 ? rest / e.count[1] : 0;
    s_origin[threadIdx.x] = (e.first[0] + 2 * i0 - 1) * K + py * ((e.first[1] + 2 * i1 - 1) * K) +
                            (DIM == 3 ? pz * ((e.first[2] + 2 * i2 - 1) * K) : 0);
  }
  __syncthreads();

  // The rows of b are on their way from the start where the registers allow it
  // (FP64 Q3 64^3 1107 -> 1029 us, Q4 3273 -> 3172; Q5 48^3 5895 -> 6271).
  constexpr bool EARLY = (K == 3 || K == 4) && PP * LINES <= NT;
  T eb[EARLY ? 2 * M : 1];
  auto rhs = [&](int t, int p) -> const T* {
    const int ln = t % LINES;
    return b + s_origin[W * (t / LINES) + p] + 1 + ln % M + (DIM == 3 ? py * (1 + ln / M) : 0) + ps;
  };
  if constexpr (EARLY) {
    const int t = (int)threadIdx.x < npair * LINES ? threadIdx.x : 0;
#pragma unroll
    for (int l = 0; l < M; ++l) {
      eb[l] = __ldg(rhs(t, 0) + ps * l);
      eb[M + l] = __ldg(rhs(t, W - 1) + ps * l);
    }
  }
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
        const T *const ua = u + s_origin[W * q] + x + pz * z, *const ub = u + s_origin[W * q + W - 1] + x + pz * z;
        E* const P = S + q * 2 * F + z * M * R + x;
        auto get = [&](int y) -> V { return PA::pack_neg(ua[py * y], ub[py * y]); };
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
        E* const P = S + t / (C * M) * 2 * F + t % (C * M) * R;
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
        const T *const ua = u + s_origin[W * q] + py * y, *const ub = u + s_origin[W * q + W - 1] + py * y;
        E* const P = S + q * 2 * F + y * R;
        closure_line<K>([&](int x) -> V { return PA::pack_neg(ua[x], ub[x]); },
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
  auto line = [&](int q, int ln) -> E* { return S + q * 2 * F + (DIM == 3 ? ln / M * R + ln % M : ln); };
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;  // 3D: x + M y; 2D: x
    const T *const ba = rhs(t, 0), *const bb = rhs(t, W - 1);
    PA::acc acc[M];
#pragma unroll
    for (int l = 0; l < M; ++l) {
      if constexpr (EARLY) acc[l] = PA::scaled(sb, PA::pack(eb[l], eb[M + l]));
      else acc[l] = PA::scaled(sb, PA::pack(__ldg(ba + ps * l), __ldg(bb + ps * l)));
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
      E* const w = S + q * 2 * F + ln % M + ln / M * M * R;
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
    E* const w = S + q * 2 * F + ln * R;
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
  const bool fresh = EXACT && mode == 0 && om == T(1);  // nothing of the old value is left
  for (int t = threadIdx.x; t < npair * LINES; t += NT) {
    const int q = t / LINES, ln = t % LINES;
    const E* const w = line(q, ln);
    V v[M];
#pragma unroll
    for (int l = 0; l < M; ++l) v[l] = PA::load(w[l * SL]);
    const bool two = W == 2 && 2 * q + 1 < nv;
    const long long ofs = 1 + ln % M + (DIM == 3 ? py * (1 + ln / M) : 0) + ps;
    T *const ga = u + s_origin[W * q] + ofs, *const gb = u + s_origin[W * q + W - 1] + ofs;
    if (EXACT && fresh) {
      pl_backward<K>(v, [&](int l, V d) {
        ga[ps * l] = PA::x(d);
        if (two) gb[ps * l] = PA::y(d);
      });
    } else {
      T oa[M], ob[M];
#pragma unroll
      for (int l = 0; l < M; ++l) {
        oa[l] = ga[ps * l];
        ob[l] = gb[ps * l];
      }
      const T keep = EXACT && mode == 0 ? T(1) - om : T(1);
      pl_backward<K>(v, [&](int l, V d) {
        ga[ps * l] = fma(om, PA::x(d), EXACT ? keep * oa[l] : oa[l]);
        if (two) gb[ps * l] = fma(om, PA::y(d), EXACT ? keep * ob[l] : ob[l]);
      });
    }
  }
}

// ---- host side ----

// Patch pairs and threads per CTA, and the CTAs per SM that the registers are
// limited for (0: left to the compiler, which then takes another schedule).  A
// pair has LINES lines in most stages, and a CTA as many pairs as fill its
// threads with them.  Measured per sweep (us), the shape taken first: FP32 Q4
// 64^3 1 pair in 64 threads 583, limited for 14 CTAs 599, 2 in 128 630, 5 in
// 256 612; Q6 40^3 with registers for 4 CTAs 552, left 615, for 1 772; FP64 Q2
// 96^3 28 in 256 758, 14 in 128 803; Q3 64^3 10 in 256 for 2 CTAs 1030, left
// 1605, 5 in 128 for 4 1265; Q5 48^3 left 5165, for 2 CTAs 5904; 2D Q7 320^2 9
// in 128 for 4 CTAs 874, left 935; Q8 320^2 8 in 128 for 4 1392, left 1783.
template <int DIM, int K>
struct ClosureCfg {
  static constexpr int M = 2 * K - 1, LINES = DIM == 3 ? M * M : M;
  static constexpr int NT = DIM == 2 || K == 1 ? 128 : DF ? 256 : K <= 3 ? 128 : K == 8 ? 256 : (LINES + 31) / 32 * 32;
  static constexpr int PP = cmax(1, std::min(NT / LINES, 48));
  static constexpr int CTAS = DIM == 2 ? (DF ? 4 : 0)
                            : DF ? (K == 3 || K == 4 || K == 7 ? 2 : 0)
                                 : (K == 4 ? 0 : K == 6 ? 4 : K >= 7 ? 2 : 1);
};

// FP64, one patch per thread (SoloDF), the same results bit for bit: shapes and
// the largest launch (patches) that takes it.  Two patches per thread halve the
// issue slots of a chip that is full; on a small colour they only lengthen each
// thread's chain, fill half of the CTAs and, on the longer lines, spill.  As many
// patches as fill the threads with the lines of the first stage.  Measured per
// sweep (us), two patches -> one, for colours of the stated patches: 3D Q1 512
// 76 -> 49 (32768: 82 -> 80); Q2 512 130 -> 66, 8000 131 -> 101 (13824: 163 ->
// 153); Q3 64 149 -> 83, 1728 154 -> 105, 8000 316 -> 299 (13824: 476 both, 10 per
// CTA 429); Q4 64 226 -> 115, 1728 271 -> 245 (2744: 312 -> 349); Q5 64 305 -> 213,
// 512 312 -> 217 (729: 312 -> 322); Q6 216 460 -> 328 (729: 677 -> 674); Q7 64 549
// -> 404 (216: 542 -> 606); Q8 216 690 -> 559, 1728 4080 -> 3279.  2D Q2 400 41 ->
// 25; Q3 262144 544 -> 460; Q5 25 115 -> 58, 25600 323 -> 263, 262144 3223 -> 2725;
// Q6 25600 447 -> 448; Q7 400 246 -> 123, 6400 271 -> 270 (9216: 317 -> 403); Q8
// 1600 306 -> 168 (3600: 314 -> 345).
template <int DIM, int K>
struct SoloCfg {
  static constexpr int C = 2 * K + 1;
  static constexpr int NT = DIM == 3 && (K == 3 || K >= 7) ? 256 : DIM == 3 && K == 4 ? 192 : 128;
  static constexpr int PP = cmax(1, NT / (DIM == 3 ? C * C : C));
  static constexpr bool ALWAYS = DIM == 2 && K <= 6;
  static constexpr int LIMIT = DIM == 2 ? (K == 7 ? 6400 : 3000)
                             : K == 1 ? 32768 : K == 2 ? 10000 : K == 3 ? 12000 : K == 5 ? 600 : K == 6 ? 1000
                             : K == 7 ? 152 : 2000;
};
// FP32 on small colours: as many threads as the first stage of a pair has lines
// in 3D from degree 5, where each pair has an SM to itself (Q5 8^3 66 -> 49, Q6 82
// -> 66, Q7 98 -> 82, Q8 115 -> 98 us a sweep), CTAs of one warp in 2D (Q3 20^2 25
// -> 17, Q6 33 -> 25, Q8 41 -> 33; equal above 1600 patches).
template <int DIM, int K>
struct SmallCfg {
  static constexpr int C = 2 * K + 1;
  static constexpr int NT = DIM == 3 ? (C * C + 31) / 32 * 32 : 32;
  static constexpr int PP = DIM == 3 ? 1 : cmax(1, 28 / C);
  static constexpr int LIMIT = DIM == 3 ? (K >= 5 ? 304 : 0) : K >= 2 ? 1600 : 0;
};

// Loads the kernel and sets its attribute, once per device.
template <int DIM, int K, int PP, int NT, int CTAS>
int closure_prepare() {
  constexpr int SMEM = ClosureSmem<DIM, K>::bytes(PP);
  static_assert(SMEM <= 227 * 1024, "sweep kernel shared memory exceeds the per-CTA limit");
  static PerDevice<bool> ready_dev;
  bool* const ready = ready_dev.get();
  if (!ready) return GMG_ERR_CUDA;
  if (!*ready) {
    auto kern = pair_closure_kernel<DIM, K, NT, PP, CTAS>;
    cudaFuncAttributes attr;
    if (cudaFuncGetAttributes(&attr, kern) != cudaSuccess ||
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM) != cudaSuccess)
      return GMG_ERR_CUDA;
    *ready = true;
  }
  return GMG_OK;
}

template <int DIM, int K, int PP, int NT, int CTAS>
int closure_launch(PatchTable& tab, const T* dinv, cudaStream_t s) {
  const int st = closure_prepare<DIM, K, PP, NT, CTAS>();
  if (st != GMG_OK) return st;
  int groups = 0;
  for (int i = 0; i < tab.n; ++i) {
    tab.e[i].group_begin = groups;
    groups += (tab.e[i].n_patches + PA::W * PP - 1) / (PA::W * PP);
  }
  tab.total_groups = groups;
  if (groups <= 0) return GMG_OK;
  pair_closure_kernel<DIM, K, NT, PP, CTAS><<<groups, NT, ClosureSmem<DIM, K>::bytes(PP), s>>>(tab, dinv);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

template <int DIM, int K>
int closure_table(PatchTable& tab, const T* dinv, int ppc, cudaStream_t s) {
  using Cfg = ClosureCfg<DIM, K>;
  // tuned patches-per-CTA variants of the batched sweep (patches come in pairs)
  if constexpr (DIM == 3 && !DF && K <= 4) {
    if (ppc == 1) return closure_launch<DIM, K, 1, 32, 1>(tab, dinv, s);
    if (ppc == 2) return closure_launch<DIM, K, 1, 64, 1>(tab, dinv, s);
    if (ppc == 4) return closure_launch<DIM, K, 2, 128, 1>(tab, dinv, s);
  }
  long long patches = 0;
  for (int i = 0; i < tab.n; ++i) patches += tab.e[i].n_patches;
  if constexpr (DF) {
    using Solo = SoloCfg<DIM, K>;
    if (Solo::ALWAYS || patches <= Solo::LIMIT)
      return launch_closure_solo(DIM, K, tab, reinterpret_cast<const double*>(dinv), s);
    if constexpr (!Solo::ALWAYS) return closure_launch<DIM, K, Cfg::PP, Cfg::NT, Cfg::CTAS>(tab, dinv, s);
  } else {
    using Small = SmallCfg<DIM, K>;
    if constexpr (Small::LIMIT > 0) {
      if (patches <= Small::LIMIT) return closure_launch<DIM, K, Small::PP, Small::NT, 0>(tab, dinv, s);
    }
    return closure_launch<DIM, K, Cfg::PP, Cfg::NT, Cfg::CTAS>(tab, dinv, s);
  }
}

}  // namespace
}  // namespace gmg
