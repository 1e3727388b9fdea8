// Shared-face form of the 3D patch sweep for FP64 problems (combined
// colourised smoother, Algorithm 4, constant coefficient, degrees 3..8), two
// faces or patches per thread in double-float arithmetic (pair_arith.cuh).
//
// The local solver is exact, so the updated interior of patch j is
// A_j^{-1} (b_j - bar A_j bar u_j^0), bar u_j^0 its closure with the interior
// set to zero (App. A.3 with eqs. "main:4", "gather", "scatter").  The
// product bar A_j bar u_j^0 involves only the closure boundary: its six
// faces.  With the two-cell 1D matrices M, K (interior rows, closure columns;
// M_I, K_I their interior columns) and the patch operator
// K (x) M (x) M + M (x) K (x) M + M (x) M (x) K (x fastest, axes x, y, z):
//   x face at closure x = f (all y, z; data v):
//     F1 = (M_y (x) M_z) v,  F2 = (K_y (x) M_z + M_y (x) K_z) v,
//     contribution K_x[:, f] (x) F1 + M_x[:, f] (x) F2;
//   y face at y = f (x interior, all z; data w):
//     G1 = (K_I,x (x) M_z + M_I,x (x) K_z) w,  G2 = (M_I,x (x) M_z) w,
//     contribution M_y[:, f] (x) G1 + K_y[:, f] (x) G2;
//   z face at z = f (x, y interior; data s):
//     H1 = (K_I,x (x) M_I,y + M_I,x (x) K_I,y) s,  H2 = (M_I,x (x) M_I,y) s,
//     contribution M_z[:, f] (x) H1 + K_z[:, f] (x) H2.
// The face between two same-colour neighbours has the same nodes and terms in
// both patches: each face plane is evaluated once per colour (face kernel)
// and read by the two patches that share it (patch kernel).  Same-colour
// patches never write each other's closure, so the faces of a colour stay
// valid while its patches are updated.
//
// What bounds both kernels is the FP32 pipe: a Dot2 term is 10 operations.
// Two patches per thread keep issue slots free for everything else: 3.6 + 1.6
// thousand warp instructions per patch (9.7 with one patch per thread), FP32
// pipe 51 % busy.  Per sweep at 64^3 (48^3): k = 3 1.12 -> 0.78 ms, k = 4 3.03 ->
// 2.13, k = 7 (48^3) 15.9 -> 11.6 with another state each pass and 9.9 repeated on
// one state: 732 bytes a thread spill there, and the local memory shares L2 with
// the vectors.
#include <algorithm>
#include <type_traits>

#include <cuda.h>
#include <cuda_runtime.h>

#include "../../include/gmg.h"
#include "async.cuh"
#include "face_geom.cuh"
#include "kernels.h"
#define GMG_PAIR_ARITH PairDF
#include "pair_lines.cuh"
#include "tma_host.h"

namespace gmg {
namespace {

constexpr int kElem = 8;  // a float pair (hi, lo) of the face buffer
__host__ __device__ constexpr int imax(int a, int b) { return a > b ? a : b; }

// ---- face kernel ----

// face pairs per CTA: enough first-stage lines for NT threads.  Shared memory
// per pair, 16-byte elements: the nodes of both faces as doubles, replaced line
// by line by the first-stage P (hi, hi, lo, lo; rows of the input length),
// then Q.
template <int K, int NT>
struct FacePairCfg {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1;
  static constexpr int PX = imax(1, NT / C), PYZ = imax(1, NT / M);
  static constexpr int SX = C * C + C * M, SY = M * C + M * M, SZ = 2 * M * M;
  static constexpr int SMEM = imax(PX * SX, PYZ * imax(SY, SZ)) * 16;
};

// CTAs [0, bx) evaluate x faces, [bx, bx + by) y faces, the rest z faces, two
// consecutive faces of a family per thread.  First stage: contract z (x and y
// faces, all closure rows) or y (z faces, interior columns); second stage:
// the remaining in-plane axis.  A line is taken one cell at a time (its two
// cells are mirror images), which halves the registers and the code.  A field
// is stored as a plane of high and a plane of low parts, each [output of the
// second stage][line], so that consecutive lanes write consecutive floats:
// F[j][l], G[i][l], H[i][j].
template <int K, int NT, int FAM>
__device__ __forceinline__ void face_family(const double* __restrict__ u, float* __restrict__ faces,
                                            const FaceGeom& fg, long long blk, float4* smem, long long* s_org) {
  using F = FacePairCfg<K, NT>;
  constexpr int C = F::C, M = F::M, LINES = M * M, FF = 2 * face_fields(K, kElem);  // floats per face
  constexpr int PER = FAM == 0 ? F::PX : F::PYZ;  // pairs per CTA
  constexpr int N1 = FAM == 0 ? C : M;            // first-stage lines per pair
  constexpr int L1 = FAM == 2 ? M : C;            // their length
  constexpr int Q1 = FAM == 2 ? 1 : 0, Q2 = FAM == 0 ? 0 : 1;  // first closure column of the stages
  const long long f0 = blk * 2 * PER;
  const int nq = (int)min((long long)2 * PER, fg.nf[FAM] - f0), np = (nq + 1) / 2;
  for (int t = threadIdx.x; t < nq; t += NT) s_org[t] = face_origin<K>(fg, FAM, f0 + t);
  __syncthreads();
  const long long s1 = FAM == 0 ? fg.py : 1;  // stride between lines
  const long long s2 = FAM == 2 ? fg.py : fg.pz;
  float4* const P = smem;  // [pair][line][L1], then [pair][line][M] of Q
  float4* const Q = smem + PER * N1 * L1;
  // gather the nodes of both faces side by side, as doubles and all in flight
  // at once (cp.async), a line per thread; x faces take the faces fastest
  // (their nodes lie a pitch apart, and neighbouring faces 2k nodes), the
  // others x
  for (int t = threadIdx.x; t < 2 * PER * N1; t += NT) {
    const int q = FAM == 0 ? t % (2 * PER) : t / N1, a = FAM == 0 ? t / (2 * PER) : t % N1;
    if (q >= nq) continue;
    const double* const src = u + s_org[q] + s1 * a;
    double* const dst = reinterpret_cast<double*>(P + ((q >> 1) * N1 + a) * L1) + (q & 1);
#pragma unroll
    for (int z = 0; z < L1; ++z) async::copy8(dst + 2 * z, src + s2 * z);
  }
  async::copy_wait_all();
  __syncthreads();
  // first stage, one line: P, Q = (M, K) v; P replaces v
  for (int t = threadIdx.x; t < np * N1; t += NT) {
    float4* const p = P + t * L1;
    float4* const q = Q + t * M;
    df2_acc ca = {{0}, {0}}, cb = {{0}, {0}};
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      df2 v[K + 1];
#pragma unroll
      for (int c = Q1; c <= K; ++c) {
        const double2 d = reinterpret_cast<const double2&>(p[r ? L1 - 1 - (c - Q1) : c - Q1]);
        v[c] = df2_make(df_from_double(d.x), df_from_double(d.y));
      }
#pragma unroll
      for (int i = 1; i < K; ++i) {
        df2_acc a, b;
        pl_cell_row<K, 0, true, Q1>(i, v, a);
        pl_cell_row<K, 1, true, Q1>(i, v, b);
        const int l = r ? M - i : i - 1;
        PA::store(p[l], df2_acc_value(a));
        PA::store(q[l], df2_acc_value(b));
      }
      pl_centre<K, 0, Q1>(r == 0, v, ca);
      pl_centre<K, 1, Q1>(r == 0, v, cb);
    }
    PA::store(p[K - 1], df2_acc_value(ca));
    PA::store(q[K - 1], df2_acc_value(cb));
  }
  __syncthreads();
  // second stage, line l of a pair: M p and K p + M q; the two-term sum is
  // the second field of x faces (F2) and the first of the others (G1, H1)
  constexpr int FA = FAM == 0 ? 0 : 2 * LINES, FB = 2 * LINES - FA;
  for (int t = threadIdx.x; t < np * M; t += NT) {
    const int pr = t / M, l = t % M;
    const float4* const p = P + pr * N1 * L1 + l;
    const float4* const q = Q + pr * N1 * M + l;
    float* const o = faces + fg.foff[FAM] * 2 + (f0 + 2 * pr) * FF + l;
    const bool two = 2 * pr + 1 < nq;
    auto put = [&](float* d, df2 v) {
      d[0] = f2_x(v.hi);
      d[LINES] = f2_x(v.lo);
      if (two) {
        d[FF] = f2_y(v.hi);
        d[FF + LINES] = f2_y(v.lo);
      }
    };
    df2_acc ca = {{0}, {0}}, cb = {{0}, {0}};
#pragma unroll 1
    for (int r = 0; r < 2; ++r) {
      df2 v[K + 1], w[K + 1];
#pragma unroll
      for (int c = Q2; c <= K; ++c) {
        const int y = r ? N1 - 1 - (c - Q2) : c - Q2;
        v[c] = PA::load(p[y * L1]);
        w[c] = PA::load(q[y * M]);
      }
#pragma unroll
      for (int i = 1; i < K; ++i) {
        df2_acc a, b;
        pl_cell_row<K, 0, true, Q2>(i, v, a);
        pl_cell_row<K, 1, true, Q2>(i, v, b);
        pl_cell_row<K, 0, false, Q2>(i, w, b);
        const int j = (r ? M - i : i - 1) * M;
        put(o + FA + j, df2_acc_value(a));
        put(o + FB + j, df2_acc_value(b));
      }
      pl_centre<K, 0, Q2>(r == 0, v, ca);
      pl_centre<K, 1, Q2>(r == 0, v, cb);
      pl_centre<K, 0, Q2>(r == 0, w, cb);
    }
    put(o + FA + (K - 1) * M, df2_acc_value(ca));
    put(o + FB + (K - 1) * M, df2_acc_value(cb));
  }
}

// (registers for 4 CTAs per SM at k = 4: 0.65 ms per 64^3 sweep, 0.69 with 5,
// 0.95 without a limit; k = 3 is faster with 6, k >= 6 with 3)
template <int K, int NT>
__global__ void __launch_bounds__(NT, K == 3 ? 6 : K <= 5 ? 4 : 3) face_pair_kernel(const double* __restrict__ u, float* __restrict__ faces,
                                                       const __grid_constant__ FaceGeom fg, int bx, int by,
                                                       int* __restrict__ next) {
  using F = FacePairCfg<K, NT>;
  extern __shared__ __align__(128) float4 face_smem[];
  __shared__ long long s_org[2 * imax(F::PX, F::PYZ)];
  const int blk = blockIdx.x;
  if (blk == 0 && threadIdx.x == 0) *next = 0;  // the patch kernel's group counter
  if (blk < bx) face_family<K, NT, 0>(u, faces, fg, blk, face_smem, s_org);
  else if (blk < bx + by) face_family<K, NT, 1>(u, faces, fg, blk - bx, face_smem, s_org);
  else face_family<K, NT, 2>(u, faces, fg, blk - bx - by, face_smem, s_org);
}

// ---- patch kernel ----

// Shared memory per patch, 8-byte elements: the interior rows of b (TMA box
// rows of XB), whose slots later hold the FD work of the pair (the two high
// parts of an entry in the first patch's slot, the low parts in the
// second's), the face blocks X0 X1 Y0 Y1 (cp.async.bulk) and the sums X0 + X1
// and Y0 + Y1 of the centre rows.  The z faces go straight to registers.
// XB = 2 mod 4 keeps a stage that walks rows at two-way conflicts.
template <int K>
struct PairSweepSmem {
  static constexpr int C = 2 * K + 1, M = 2 * K - 1;
  static constexpr int XB0 = (M + 1 + 1 + 1) / 2 * 2;  // M + 1 nodes after the alignment shift, even
  static constexpr int XB = XB0 % 4 == 2 ? XB0 : XB0 + 2;
  static constexpr int NB = (M * M * XB + 15) / 16 * 16;  // boxes start on 128 bytes
  static constexpr int FS = face_fields(K, kElem);
  static constexpr int PATCH = (NB + 6 * FS + 15) / 16 * 16;
  static constexpr int BOX_BYTES = M * M * XB * 8, FACE_BYTES = FS * 8;
};

struct PairSweepArgs {
  double* u;
  const float* faces;
  const float2* dinv;  // float pairs
  int* next;  // groups handed out beyond the first of each CTA (zeroed by the face kernel)
  int* err;
  long long py, pz;
  int first[3], count[3];
  int n_patches, ngroups;
  long long foff[3];
  double omega;
  float sb;      // h^{2-d} = n, exact in float
  int undamped;  // omega == 1
};

// One colour of the sweep: persistent CTAs take groups of 2 PP consecutive
// patches, a thread carries the same line of patches 2q and 2q + 1.  Per
// patch one lane issues a TMA box of b and four bulk copies of its x and y
// faces, all of a group completing on one mbarrier (bounded wait; an expired
// wait sets err and the kernel carries on).  Stages, each on lines of one axis:
//   z: r = h^{2-d} b - (face terms), forward transform
//   y: forward | x: forward, diagonal, backward | y: backward
//   z: backward, u = omega d + (1 - omega) u_old
// The first and last stage run along z so that the lanes of a warp hold
// consecutive x: loads and stores of u touch whole sectors.  The face blocks
// are free after the first stage: the next group's faces are copied there
// during the transforms.
template <int K, int NT, int PP, int CTAS>
__global__ void __launch_bounds__(NT, CTAS) pair_sweep_kernel(const __grid_constant__ PairSweepArgs fa,
                                                              const __grid_constant__ CUtensorMap bmap) {
  using Z = PairSweepSmem<K>;
  constexpr int M = Z::M, XB = Z::XB, FS = Z::FS, LINES = M * M, NP = 2 * PP;
  static_assert(NP <= NT, "one lane issues the copies of one patch");
  constexpr int PASSES = (PP * LINES + NT - 1) / NT;  // lines per thread and stage
  // Idle threads repeat line 0 up to k = 4: control flow stays uniform and the
  // coefficients come through uniform registers.  Above, ptxas then keeps so
  // many coefficients that the lines spill (k = 7: 15.5 against 7.8 ms).
  constexpr bool UNI = K <= 4;
  extern __shared__ __align__(128) unsigned char smem_raw[];
  double* const S = reinterpret_cast<double*>(smem_raw + ((128 - (async::smem_u32(smem_raw) & 127)) & 127));
  __shared__ long long s_origin[NP], s_zface[NP][2];  // closure origin, float offsets of the z faces
  __shared__ float4 s_edge[M];                        // end column of row i: -M (hi, lo), -K (hi, lo)
  __shared__ int s_next;
  __shared__ __align__(8) uint64_t s_bar;
  uint32_t phase = 0;
  bool wait_ok = true;
  const int cx = fa.count[0], cy = fa.count[1];
  if (threadIdx.x == 0) async::mbar_init(&s_bar, 1);
  for (int i = threadIdx.x; i < M; i += NT) {
    const float4 m = p_E[pl_off_end(K) + 2 * i], s = p_E[pl_off_end(K) + 2 * i + 1];
    s_edge[i] = make_float4(m.x, m.z, s.x, s.z);
  }
  // x offset of the interior inside the TMA box, the same for every patch of
  // the colour: closure origins in x differ by multiples of 2K
  const int sh = ((fa.first[0] - 1) * K) % 2 + 1;
  __syncthreads();

  // Copies of a group: the patches are spread over the warps, as a warp issues
  // its lanes' copies one after the other (ten patches' by one warp took 10 %
  // of a group's time).
  const int fq = threadIdx.x / 32 + (threadIdx.x % 32) * (NT / 32);  // the patch this thread copies
  auto position = [&](int pid, int& ix, int& iy, int& iz) {
    ix = pid % cx;
    const int rest = pid / cx;
    iy = rest % cy;
    iz = rest / cy;
  };
  auto fetch_faces = [&](int grp) {
    const int pid = grp * NP + fq;
    if (fq >= NP || pid >= fa.n_patches) return;
    int ix, iy, iz;
    position(pid, ix, iy, iz);
    const long long fxi = ((long long)iz * cy + iy) * (cx + 1) + ix, fyi = ((long long)iz * (cy + 1) + iy) * cx + ix;
    const long long face[4] = {fa.foff[0] + fxi * FS, fa.foff[0] + (fxi + 1) * FS, fa.foff[1] + fyi * FS,
                               fa.foff[1] + (fyi + cx) * FS};
#pragma unroll
    for (int f = 0; f < 4; ++f)
      async::bulk_load(S + fq * Z::PATCH + Z::NB + f * FS, fa.faces + 2 * face[f], Z::FACE_BYTES, &s_bar);
  };
  // b, and the origins; the group's one arrival announces all of its bytes
  auto fetch_b = [&](int grp) {
    if (threadIdx.x == 0)
      async::mbar_arrive_expect_tx(&s_bar, (uint32_t)(min(NP, fa.n_patches - grp * NP) * (Z::BOX_BYTES + 4 * Z::FACE_BYTES)));
    const int pid = grp * NP + fq;
    if (fq >= NP || pid >= fa.n_patches) return;
    int ix, iy, iz;
    position(pid, ix, iy, iz);
    const int o0 = (fa.first[0] + 2 * ix - 1) * K, o1 = (fa.first[1] + 2 * iy - 1) * K,
              o2 = (fa.first[2] + 2 * iz - 1) * K;
    s_origin[fq] = o0 + fa.py * o1 + fa.pz * o2;
    const long long fzi = ((long long)iz * cy + iy) * cx + ix;
    s_zface[fq][0] = 2 * (fa.foff[2] + fzi * FS);
    s_zface[fq][1] = 2 * (fa.foff[2] + (fzi + (long long)cy * cx) * FS);
    async::tma_load_3d(S + fq * Z::PATCH, &bmap, o0 - o0 % 2, o1 + 1, o2 + 1, &s_bar);
  };

  int grp = blockIdx.x;
  if (grp < fa.ngroups) {
    fetch_faces(grp);
    fetch_b(grp);
  }
  __syncthreads();
  while (grp < fa.ngroups) {
    // the next group: whichever CTA gets there first takes it (with a fixed
    // share per CTA the SMs finish a Q4 64^3 colour between 132 and 187 us)
    int next = 0;
    if (threadIdx.x == 0) next = gridDim.x + atomicAdd(fa.next, 1);
    const int nv = min(NP, fa.n_patches - grp * NP), npair = (nv + 1) / 2;
    // z faces H1[i][j], H2[i][j] of both ends of this thread's first-stage
    // lines, from global memory: on their way during the sums
    float ha[PASSES][8], hb[PASSES][8];  // [end][field][high, low] of both patches
#pragma unroll
    for (int ps = 0; ps < PASSES; ++ps) {
      const int t = threadIdx.x + ps * NT < npair * LINES ? threadIdx.x + ps * NT : 0;
      const int q = t / LINES, ln = t % LINES, o = ln % M * M + ln / M;
      const int qb = 2 * q + 1 < nv ? 2 * q + 1 : 2 * q;  // a lone last patch is carried twice
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        ha[ps][e] = __ldcg(fa.faces + s_zface[2 * q][e / 4] + o + e % 4 * LINES);
        hb[ps][e] = __ldcg(fa.faces + s_zface[qb][e / 4] + o + e % 4 * LINES);
      }
    }
    if (wait_ok && !async::mbar_wait(&s_bar, phase)) wait_ok = false;
    phase ^= 1u;

    // ---- sums of the x and of the y faces, for the centre rows: column 0 of
    // the two-cell matrices is nonzero on rows 0..K-1 and column 2K on rows
    // K-1..M-1, and on row K-1 (the vertex row) both hold the same entry, so a
    // face term there is that entry times the sum of the two faces' fields ----
    for (int t = threadIdx.x; t < npair * 4 * LINES; t += NT) {
      const int q = t / (4 * LINES), e = t % (4 * LINES);  // e: axis, field, entry
      const int o = (e / LINES) * 2 * LINES + e % LINES;    // its high part among the sums
      float* const a = reinterpret_cast<float*>(S + 2 * q * Z::PATCH + Z::NB);
      const float* const p = a + o + (o >= 2 * FS ? 2 * FS : 0);  // X0 or Y0
      auto both = [&](int f) -> df2 {
        return {f2_make(p[f], p[f + 2 * Z::PATCH]), f2_make(p[f + LINES], p[f + LINES + 2 * Z::PATCH])};
      };
      const df2 v = df2_add(both(0), both(2 * FS));
      float* const d = a + 8 * FS + o;
      d[0] = f2_x(v.hi);
      d[LINES] = f2_x(v.lo);
      d[2 * Z::PATCH] = f2_y(v.hi);
      d[2 * Z::PATCH + LINES] = f2_y(v.lo);
    }
    __syncthreads();

    // ---- residual on interior z line (i, j), forward transform along z ----
#pragma unroll
    for (int ps = 0; ps < PASSES; ++ps) {
      const bool on = threadIdx.x + ps * NT < npair * LINES;
      if (!UNI && !on) break;
      const int t = on ? threadIdx.x + ps * NT : 0;
      const int q = t / LINES, ln = t % LINES, i = ln % M, j = ln / M;
      double* const A = S + 2 * q * Z::PATCH;
      // face value of both patches whose high part is float o of a patch's face blocks
      const float* const FA = reinterpret_cast<const float*>(A + Z::NB);
      auto face = [&](int o) -> df2 {
        return {f2_make(FA[o], FA[o + 2 * Z::PATCH]), f2_make(FA[o + LINES], FA[o + LINES + 2 * Z::PATCH])};
      };
      auto zface = [&](int e) -> df2 {
        return {f2_make(ha[ps][e], hb[ps][e]), f2_make(ha[ps][e + 1], hb[ps][e + 1])};
      };
      const float4 ex = s_edge[i], ey = s_edge[j];
      const df2_coef mx = {f2_dup(ex.x), f2_dup(ex.y)}, kx = {f2_dup(ex.z), f2_dup(ex.w)};
      const df2_coef my = {f2_dup(ey.x), f2_dup(ey.y)}, ky = {f2_dup(ey.z), f2_dup(ey.w)};
      const int fx = 2 * FS * (i < K - 1 ? 0 : i > K - 1 ? 1 : 4) + j * M;
      const int fy = 2 * FS * (j < K - 1 ? 2 : j > K - 1 ? 3 : 5) + i * M;
      const f2 sb = f2_dup(fa.sb);
      df2 r[M];
#pragma unroll
      for (int l = 0; l < M; ++l) {
        const double* const p = A + (l * M + j) * XB + sh + i;
        df2_acc acc = df2_acc_scaled(sb, df2_make(df_from_double(p[0]), df_from_double(p[Z::PATCH])));
        df2_acc_add(acc, kx, face(fx + l));
        df2_acc_add(acc, mx, face(fx + 2 * LINES + l));
        df2_acc_add(acc, ky, face(fy + 2 * LINES + l));
        df2_acc_add(acc, my, face(fy + l));
        const df2_coef mz = pl_coef(p_E[pl_off_end(K) + 2 * l]), kz = pl_coef(p_E[pl_off_end(K) + 2 * l + 1]);
        if (l <= K - 1) {
          df2_acc_add(acc, kz, zface(2));
          df2_acc_add(acc, mz, zface(0));
        }
        if (l >= K - 1) {
          df2_acc_add(acc, kz, zface(6));
          df2_acc_add(acc, mz, zface(4));
        }
        r[l] = df2_acc_value(acc);
      }
      f2* const Wh = reinterpret_cast<f2*>(A) + j * XB + sh + i;
      f2* const Wl = Wh + Z::PATCH;
      pl_forward<K>(r, [&](int l, df2 v) {
        if (on) {
          Wh[l * M * XB] = v.hi;
          Wl[l * M * XB] = v.lo;
        }
      });
    }
    if (threadIdx.x == 0) s_next = next;
    async::fence_proxy_async();  // reads of the faces before the next copies write them
    __syncthreads();
    grp = s_next;
    if (grp < fa.ngroups) fetch_faces(grp);
    // ---- local solve by fast diagonalisation (App. A.3), in place ----
    auto line_y = [&](auto forward) {
#pragma unroll 1
      for (int ps = 0; ps < PASSES; ++ps) {
        const bool on = threadIdx.x + ps * NT < npair * LINES;
        if (!UNI && !on) break;
        const int t = on ? threadIdx.x + ps * NT : 0;
        const int q = t / LINES, ln = t % LINES, i = ln % M, l = ln / M;
        f2* const Wh = reinterpret_cast<f2*>(S + 2 * q * Z::PATCH) + l * M * XB + sh + i;
        f2* const Wl = Wh + Z::PATCH;
        df2 v[M];
#pragma unroll
        for (int j = 0; j < M; ++j) v[j] = {Wh[j * XB], Wl[j * XB]};
        auto put = [&](int j, df2 x) {
          if (on) {
            Wh[j * XB] = x.hi;
            Wl[j * XB] = x.lo;
          }
        };
        if constexpr (decltype(forward)::value) pl_forward<K>(v, put);
        else pl_backward<K>(v, put);
      }
    };
    line_y(std::true_type());
    __syncthreads();
#pragma unroll 1
    for (int ps = 0; ps < PASSES; ++ps) {
      const bool on = threadIdx.x + ps * NT < npair * LINES;
      if (!UNI && !on) break;
      const int t = on ? threadIdx.x + ps * NT : 0;
      const int q = t / LINES, ln = t % LINES;  // ln = j + M l
      f2* const Wh = reinterpret_cast<f2*>(S + 2 * q * Z::PATCH) + ln * XB + sh;
      f2* const Wl = Wh + Z::PATCH;
      // the diagonal is symmetric in its three indices: entry (j, l, i), so
      // that consecutive lanes read consecutive pairs
      auto scaled = [&](int i, df2 z) -> df2 {
        const float2 d = __ldg(fa.dinv + i * LINES + ln);
        return df2_acc_value(df2_acc_first({f2_dup(d.x), f2_dup(d.y)}, z));
      };
      auto put = [&](int i, df2 z) {
        if (on) {
          Wh[i] = z.hi;
          Wl[i] = z.lo;
        }
      };
      df2 v[M];
#pragma unroll
      for (int i = 0; i < M; ++i) v[i] = {Wh[i], Wl[i]};
      if constexpr (K <= 6) {
        df2 x[M];
        pl_forward<K>(v, [&](int i, df2 z) { x[i] = scaled(i, z); });
        pl_backward<K>(x, put);
      } else {  // two lines in registers would spill: through this thread's line in shared memory
        pl_forward<K>(v, [&](int i, df2 z) { put(i, scaled(i, z)); });
        asm volatile("" ::: "memory");
#pragma unroll
        for (int i = 0; i < M; ++i) v[i] = {Wh[i], Wl[i]};
        pl_backward<K>(v, put);
      }
    }
    __syncthreads();
    line_y(std::false_type());
    __syncthreads();
    // ---- backward along z and scatter (eq. "scatter"); undamped steps write
    // the new value without reading the old one ----
    auto scatter = [&](auto damped) {
#pragma unroll 1
      for (int ps = 0; ps < PASSES; ++ps) {
        const bool on = threadIdx.x + ps * NT < npair * LINES;
        if (!UNI && !on) break;
        const int t = on ? threadIdx.x + ps * NT : 0;
        const int q = t / LINES, ln = t % LINES, i = ln % M, j = ln / M;
        const f2* const Wh = reinterpret_cast<const f2*>(S + 2 * q * Z::PATCH) + j * XB + sh + i;
        const f2* const Wl = Wh + Z::PATCH;
        df2 v[M];
#pragma unroll
        for (int l = 0; l < M; ++l) v[l] = {Wh[l * M * XB], Wl[l * M * XB]};
        const bool two = on && 2 * q + 1 < nv;
        const long long ofs = (1 + i) + fa.py * (1 + j) + fa.pz;
        double* const ua = fa.u + s_origin[2 * q] + ofs;
        double* const ub = fa.u + s_origin[2 * q + 1 < nv ? 2 * q + 1 : 2 * q] + ofs;
        pl_backward<K>(v, [&](int l, df2 x) {
          double da = df_to_double(df2_x(x)), db = df_to_double(df2_y(x));
          if constexpr (decltype(damped)::value) {
            da = fma(fa.omega, da, (1.0 - fa.omega) * ua[fa.pz * l]);
            db = fma(fa.omega, db, (1.0 - fa.omega) * ub[fa.pz * l]);
          }
          if (on) ua[fa.pz * l] = da;
          if (two) ub[fa.pz * l] = db;
        });
      }
    };
    if (fa.undamped) scatter(std::false_type());
    else scatter(std::true_type());
    async::fence_proxy_async();  // accesses of the work before the next b is copied there
    __syncthreads();
    if (grp < fa.ngroups) fetch_b(grp);
    __syncthreads();
  }
  if (!wait_ok) atomicExch(fa.err, GMG_ERR_TIMEOUT);
}

// ---- host side ----

// Patch pairs and threads per CTA, and the CTAs per SM that the registers are
// limited for.  PP fills the threads with lines (k = 4: 245 of 256); more,
// smaller CTAs lose lanes, more registers lose warps.  Measured per 64^3
// sweep at k = 4 (both kernels): 2.16 ms with 5 pairs, 256 threads, 2 CTAs;
// 2.33 with 3, 160, 3; 2.55 with 2, 128, 4; 3.1 with one CTA per SM.  Meshes
// down to 16^3 keep the same shape (213 us a sweep; 197 with one pair per CTA).
template <int K>
struct PairSweepCfg {
  static constexpr int PP = K <= 4 ? 5 : K == 5 ? 3 : 1;
  static constexpr int NT = K == 3 || K == 6 ? 128 : K == 7 ? 192 : 256;
  static constexpr int CTAS = K == 3 ? 4 : K == 8 ? 1 : 2;
  static constexpr int SMEM = 2 * PP * PairSweepSmem<K>::PATCH * 8 + 128;
  static_assert(SMEM <= 227 * 1024, "shared-face sweep exceeds the shared memory of a CTA");
};
constexpr int kFaceThreads = 128;

// At degrees 5 to 7 a colour of at most this many patches, while each patch has an
// SM to itself, goes to the coarse-level kernel, one output per thread (us a sweep
// of 6^3: Q5 289 -> 115, Q6 345 -> 181, Q7 489 -> 289).  Not at degree 8 (625 : 421):
// its error against 64 bits is a quarter larger there, as it evaluates the
// residual on the whole closure and not on its boundary (8^3: 2.5e-14 against
// 2.0e-14; Q5 1.08e-14 and 1.05e-14, Q6 1.8e-14 and 1.9e-14, Q7 2.3e-14 and 3.0e-14).
constexpr int kFewPatches = 128;

template <typename KernelT>
int opt_in(KernelT kern, int smem) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) == cudaSuccess ? GMG_OK
                                                                                                     : GMG_ERR_CUDA;
}

template <int K>
int face_sweep(const PatchLaunch& pl, double* u, const double* b, const double* dinv, double* faces, cudaStream_t s) {
  constexpr int FNT = kFaceThreads;
  using FC = FacePairCfg<K, FNT>;
  using SC = PairSweepCfg<K>;
  using Z = PairSweepSmem<K>;
  auto fk = face_pair_kernel<K, FNT>;
  auto pk = pair_sweep_kernel<K, SC::NT, SC::PP, SC::CTAS>;
  static PerDevice<int> slots_dev;  // resident CTAs of the patch kernel
  int* const slots = slots_dev.get();
  if (!slots) return GMG_ERR_CUDA;
  if (*slots == 0) {
    int per_sm = 0, sms = 0;
    if (opt_in(fk, FC::SMEM) != GMG_OK || opt_in(pk, SC::SMEM) != GMG_OK) return GMG_ERR_CUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, pk, SC::NT, SC::SMEM) != cudaSuccess || per_sm <= 0 ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, current_device()) != cudaSuccess || sms <= 0)
      return GMG_ERR_CUDA;
    *slots = per_sm * sms;
  }
  const FaceGeom fg = face_geom(pl, kElem);
  const long long bx = (fg.nf[0] + 2 * FC::PX - 1) / (2 * FC::PX), by = (fg.nf[1] + 2 * FC::PYZ - 1) / (2 * FC::PYZ),
                  bz = (fg.nf[2] + 2 * FC::PYZ - 1) / (2 * FC::PYZ);
  if (bx + by + bz > (1LL << 31) - 1) return GMG_ERR_UNSUPPORTED;
  // the buffer begins with the group counter (16 bytes), then the faces
  int* const next = reinterpret_cast<int*>(faces);
  float* const fbuf = reinterpret_cast<float*>(faces + 2);
  fk<<<(unsigned)(bx + by + bz), FNT, FC::SMEM, s>>>(u, fbuf, fg, (int)bx, (int)by, next);
  count_launch();
  if (cudaGetLastError() != cudaSuccess) return GMG_ERR_CUDA;

  const int m = 2 * K - 1;
  PairSweepArgs fa;
  fa.u = u;
  fa.faces = fbuf;
  fa.dinv = reinterpret_cast<const float2*>(dinv + m * m * m);
  fa.next = next;
  fa.err = device_wait_flag();
  if (!fa.err) return GMG_ERR_CUDA;
  fa.py = pl.g.py;
  fa.pz = pl.g.pz;
  for (int a = 0; a < 3; ++a) {
    fa.first[a] = pl.first[a];
    fa.count[a] = pl.count[a];
    fa.foff[a] = fg.foff[a];
  }
  fa.n_patches = pl.n_patches;
  fa.ngroups = (pl.n_patches + 2 * SC::PP - 1) / (2 * SC::PP);
  fa.sb = (float)pl.sb;
  fa.omega = pl.omega;
  fa.undamped = pl.omega == 1.0;
  CUtensorMap bmap;
  if (!tma_encode(&bmap, b, 8, 3, pl.g.N, pl.g.py, pl.g.pz, Z::XB, Z::M)) return GMG_ERR_CUDA;
  pk<<<std::min(fa.ngroups, *slots), SC::NT, SC::SMEM, s>>>(fa, bmap);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

}  // namespace

int upload_pair_sweep_tables(int k, const double* Mp, const double* Kp, const double* That) {
  if (k < 3 || k > 8) return GMG_OK;  // the form starts at degree 3
  return pl_upload(k, Mp, Kp, That);
}

template <>
int launch_patch_faces<double>(const PatchLaunch& pl, double* u, const double* b, const double* dinv, double* faces,
                               cudaStream_t s) {
  if (pl.g.dim != 3 || pl.g.k < 3 || pl.g.k > 8 || pl.mode != 0 || pl.plist || !faces) return GMG_ERR_UNSUPPORTED;
  if (!tma_vector_ok(b, 8, 3, pl.g.py, pl.g.pz)) return GMG_ERR_UNSUPPORTED;
  if (pl.n_patches <= 0) return GMG_OK;
  if (pl.g.k >= 5 && pl.g.k <= 7 && pl.n_patches <= kFewPatches) return launch_patch_small<double>(pl, u, b, dinv, s);
  switch (pl.g.k) {
    case 3: return face_sweep<3>(pl, u, b, dinv, faces, s);
    case 4: return face_sweep<4>(pl, u, b, dinv, faces, s);
    case 5: return face_sweep<5>(pl, u, b, dinv, faces, s);
    case 6: return face_sweep<6>(pl, u, b, dinv, faces, s);
    case 7: return face_sweep<7>(pl, u, b, dinv, faces, s);
    default: return face_sweep<8>(pl, u, b, dinv, faces, s);
  }
}

template <>
long long face_buffer_elems<double>(const PatchLaunch& pl) {
  return 2 + face_buffer_total(pl, kElem);  // the group counter, then the faces
}

}  // namespace gmg
