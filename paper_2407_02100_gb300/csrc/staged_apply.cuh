// FP64 form of the 3D level operator in three passes, one per axis, each a 1D
// contraction with the global 1D matrices (unit-cell mass M and stiffness K
// assembled along one axis), through two workspace vectors:
//   pass z: P = M_z u,  Q = K_z u
//   pass y: A1 = M_y P, A2 = K_y P + M_y Q
//   pass x: y = alpha (K_x A1 + M_x A2) + beta b     (interior nodes)
// which is A = K (x) M (x) M + M (x) K (x) M + M (x) M (x) K by sum
// factorisation (Sec. 2, App. A.1 with the cell integrals summed into
// global rows).  The tile kernel recomputes a halo of up to K + 1 nodes per
// direction in its first two stages; here only the y rows of a tile's left
// columns are evaluated twice, for six passes of level vectors through HBM.
// Included by patch_f64.cu after patch_kernels.cuh (T = double).
#pragma once

namespace gmg {
namespace GMG_NS {

// A thread evaluates the K global rows of nodes c K .. c K + K - 1 along an
// axis (cell c of that axis) from the 2K + 1 inputs c K - K .. c K + K (zero
// outside the lattice).  Row c K (a vertex) is row K of cell c - 1 plus row 0
// of cell c; row c K + p (0 < p < K) is row p of cell c.
//
// acc += (FIRST: =) global row p of a segment (row c K + p, see above), matrix
// KIND, applied to the 2K + 1 window v, in double-float (Dot2)
template <int K, int KIND, bool FIRST>
__device__ __forceinline__ void segment_row_df(int p, const dfv (&v)[2 * K + 1], df_acc& acc) {
  auto eh = [](int r, int q) { return KIND == 0 ? c_Mchi[off_cell(K) + r * (K + 1) + q] : c_Kchi[off_cell(K) + r * (K + 1) + q]; };
  auto el = [](int r, int q) { return KIND == 0 ? c_Mclo[off_cell(K) + r * (K + 1) + q] : c_Kclo[off_cell(K) + r * (K + 1) + q]; };
  if (p == 0) {
#pragma unroll
    for (int q = 0; q <= K; ++q) {
      if (FIRST && q == 0) acc = df_acc_first(eh(K, q), el(K, q), v[q]);
      else df_acc_add(acc, eh(K, q), el(K, q), v[q]);
    }
  }
#pragma unroll
  for (int q = 0; q <= K; ++q) {
    if (FIRST && p > 0 && q == 0) acc = df_acc_first(eh(p, q), el(p, q), v[K + q]);
    else df_acc_add(acc, eh(p, q), el(p, q), v[K + q]);
  }
}

// The same in double-float arithmetic (FP64 problems; GB300 runs FP64 at about
// 1/74 of its FP32 rate), in two launches: the workspace vectors hold float
// pairs (hi, lo) in the 8 bytes of a double, the rows accumulate in Dot2 form
// with the float-pair cell matrices, and alpha (K A1 + M A2) + beta b is formed
// in FP64 from the pair's value (two FP64 operations per node).
//
// Pass z.  A CTA takes 128 consecutive x positions of one y and one cell layer.
template <int K>
__global__ void __launch_bounds__(128) pass_z_df_kernel(const double* __restrict__ in, float2* __restrict__ P,
                                                        float2* __restrict__ Q, const LevelGeom g) {
  constexpr int W = 2 * K + 1;
  const int N = g.N;
  const long long py = g.py, pz = g.pz;
  const long long t = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (long long)N * N * g.n) return;
  const int x = (int)(t % N);
  const long long r = t / N;
  const int y = (int)(r % N), c = (int)(r / N);
  const long long base = x + py * y + pz * ((long long)c * K - K);
  dfv a[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    const bool ok = w >= K || c > 0;
    a[w] = ok ? df_from_double(in[base + pz * w]) : dfv{0.f, 0.f};
  }
#pragma unroll
  for (int p = 0; p < K; ++p) {
    if (p == 0 && c == 0) continue;  // a Dirichlet node
    const long long o = base + pz * (K + p);
    df_acc r0, r1;
    segment_row_df<K, 0, true>(p, a, r0);
    segment_row_df<K, 1, true>(p, a, r1);
    const dfv v0 = df_acc_value(r0), v1 = df_acc_value(r1);
    P[o] = make_float2(v0.hi, v0.lo);
    Q[o] = make_float2(v1.hi, v1.lo);
  }
}

// Passes y and x together on a tile of BX x BY cells of one z plane: A1 and A2
// of the tile (with the K + 1 columns to its left) stay in shared memory, so
// that four of the ten passes over level vectors are not made: Q4 64^3 403 ->
// 368 us with pass z (140 us), Q3 51^3 108 -> 91.  Both launches are bound by the
// FP32 pipe (Dot2 terms of 10 operations); limits on the registers only made
// them slower (Q4 3 CTAs per SM 403 us, Q7 32^3 2 CTAs 509 against 444 with 9-cell tiles).  The y
// rows are evaluated for ((BX + 1) K + 1) / (BX K) of the columns that are needed.
template <int K>
struct PlanePass {
  // the widest tile whose columns with their halo, 4 cells high, take one round
  // of the threads (Q7 48^3 1449 -> 1179 us, Q3 51^3 102 -> 91, against 64 / K
  // cells); at K = 4 16 cells: a quarter faster than 14 where they save a tile (Q4
  // 16^3 15.7 : 19.7 us, 32^3 52 : 66, 44^3 134 : 154, 64^3 365 : 406), up to 2.5 %
  // slower elsewhere (28^3 equal, 42^3 124 : 121, 56^3 267 : 261)
  static constexpr int BX = K == 4 ? 16 : (63 - K) / K, BY = 4, NT = 256;
  static constexpr int EX = (BX + 1) * K + 1, EY = BY * K;
  static constexpr int EXP = EX | 1;  // odd row: lanes of the x stage lie K entries apart
  static constexpr int BYTES = 2 * EY * EXP * (int)sizeof(float2);
};

template <int K>
__global__ void __launch_bounds__(PlanePass<K>::NT) pass_yx_df_kernel(
    const float2* __restrict__ P, const float2* __restrict__ Q, double* __restrict__ yout,
    const double* __restrict__ bvec, const LevelGeom g, double alpha, double beta, int tx, int ty) {
  using D = PlanePass<K>;
  constexpr int BX = D::BX, BY = D::BY, EX = D::EX, EXP = D::EXP, NT = D::NT, W = 2 * K + 1;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float2* const A1 = reinterpret_cast<float2*>(smem_raw);
  float2* const A2 = A1 + D::EY * EXP;
  const int N = g.N, n = g.n;
  const long long py = g.py;
  const int t0 = blockIdx.x % tx, t1 = blockIdx.x / tx % ty, z = 1 + blockIdx.x / (tx * ty);
  const long long plane = g.pz * z;
  const int x0 = (t0 * BX - 1) * K, c1 = t1 * BY;
  for (int t = threadIdx.x; t < EX * BY; t += NT) {
    const int xi = t % EX, x = x0 + xi, cy = t / EX, c = c1 + cy;
    const bool in = x >= 0 && x < N && c < n;
    const long long base = plane + x + py * ((long long)c * K - K);
    dfv a[W], b[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const bool ok = in && (w >= K || c > 0);
      const float2 va = ok ? P[base + py * w] : make_float2(0.f, 0.f);
      const float2 vb = ok ? Q[base + py * w] : make_float2(0.f, 0.f);
      a[w] = {va.x, va.y};
      b[w] = {vb.x, vb.y};
    }
#pragma unroll
    for (int p = 0; p < K; ++p) {
      df_acc r0, r1;
      segment_row_df<K, 0, true>(p, a, r0);
      segment_row_df<K, 1, true>(p, a, r1);
      segment_row_df<K, 0, false>(p, b, r1);
      const dfv v0 = df_acc_value(r0), v1 = df_acc_value(r1);
      const int o = (cy * K + p) * EXP + xi;
      A1[o] = make_float2(v0.hi, v0.lo);
      A2[o] = make_float2(v1.hi, v1.lo);
    }
  }
  __syncthreads();
  // one thread per cell of a row, rows along the lanes (odd row stride); the
  // results go back through shared memory, so that the rows of b and y are
  // read and written with lanes along x
  static_assert(BX * D::EY <= NT, "one thread per cell row");
  const int r = threadIdx.x % D::EY, cx = threadIdx.x / D::EY;
  dfv v[K];
  if (cx < BX) {
    dfv a[W], b[W];
#pragma unroll
    for (int w = 0; w < W; ++w) {
      const float2 va = A1[r * EXP + cx * K + w], vb = A2[r * EXP + cx * K + w];
      a[w] = {va.x, va.y};
      b[w] = {vb.x, vb.y};
    }
#pragma unroll
    for (int p = 0; p < K; ++p) {
      df_acc acc;
      segment_row_df<K, 1, true>(p, a, acc);
      segment_row_df<K, 0, false>(p, b, acc);
      v[p] = df_acc_value(acc);
    }
  }
  __syncthreads();
  if (cx < BX) {
#pragma unroll
    for (int p = 0; p < K; ++p) A1[r * EXP + cx * K + p] = make_float2(v[p].hi, v[p].lo);
  }
  __syncthreads();
  for (int t = threadIdx.x; t < BX * K * D::EY; t += NT) {
    const int xi = t % (BX * K), yr = t / (BX * K), x = x0 + K + xi, y = c1 * K + yr;
    if (x < 1 || x > N - 2 || y < 1 || y > N - 2) continue;
    const float2 f = A1[yr * EXP + xi];
    const long long o = plane + py * y + x;
    double d = alpha * df_to_double(dfv{f.x, f.y});
    if (bvec) d = fma(beta, bvec[o], d);
    yout[o] = d;
  }
}

template <int K>
static int staged_apply_impl(const ApplyLaunch& al, const double* x, double* y, const double* bvec, cudaStream_t s) {
  using D = PlanePass<K>;
  static_assert(D::BYTES <= 48 * 1024, "tile exceeds the default shared memory of a CTA");
  const LevelGeom& g = al.g;
  float2* const P = static_cast<float2*>(al.ws);
  float2* const Q = P + g.pz * g.N;
  const long long N = g.N, tx = (g.n + D::BX - 1) / D::BX, ty = (g.n + D::BY - 1) / D::BY;
  pass_z_df_kernel<K><<<(unsigned)((N * N * g.n + 127) / 128), 128, 0, s>>>(x, P, Q, g);
  pass_yx_df_kernel<K><<<(unsigned)(tx * ty * (N - 2)), D::NT, D::BYTES, s>>>(P, Q, y, bvec, g, al.alpha, al.beta,
                                                                              (int)tx, (int)ty);
  count_launch(2);
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

}  // namespace GMG_NS
}  // namespace gmg
