// Closure form of the patch sweep in single precision.
#define GMG_PAIR_ARITH PairF32
#include "pair_closure.cuh"

namespace gmg {
namespace {

template <int DIM, int K>
int table_launches(const PatchLaunch* pls, T* const* us, const T* const* bs, int n, const T* dinv, int ppc,
                   cudaStream_t s) {
  for (int i0 = 0; i0 < n; i0 += kMaxTable) {
    PatchTable tab;
    tab.n = 0;
    tab.mode = pls[i0].mode;
    tab.omega = pls[i0].omega;
    for (int i = i0; i < std::min(n, i0 + kMaxTable); ++i)
      if (pls[i].n_patches > 0) fill_entry(tab.e[tab.n++], pls[i], us[i], bs[i]);
    if (tab.n == 0) continue;
    const int st = closure_table<DIM, K>(tab, dinv, ppc, s);
    if (st != GMG_OK) return st;
  }
  return GMG_OK;
}

}  // namespace

template <>
int upload_closure_tables<float>(int k, const double* Mp, const double* Kp, const double* That) {
  return pl_upload(k, Mp, Kp, That);
}

template <>
int launch_patch_table<float>(int dim, int k, const PatchLaunch* pls, float* const* us, const float* const* bs, int n,
                             const float* dinv, int ppc, cudaStream_t s) {
  GMG_DISPATCH(table_launches, dim, k, pls, us, bs, n, dinv, ppc, s)
}

template <>
int launch_patch_colour<float>(const PatchLaunch& pl, float* u, const float* b, const float* dinv, cudaStream_t s) {
  return launch_patch_table<float>(pl.g.dim, pl.g.k, &pl, &u, &b, 1, dinv, 0, s);
}

}  // namespace gmg
