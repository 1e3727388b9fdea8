// Closure form of the patch sweep in double precision.
#define GMG_PAIR_ARITH PairDF
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

// both kernels of a degree: a launch takes one or the other by its patches
template <int DIM, int K>
int prepare_all() {
  using Cfg = ClosureCfg<DIM, K>;
  if constexpr (!SoloCfg<DIM, K>::ALWAYS) {
    const int st = closure_prepare<DIM, K, Cfg::PP, Cfg::NT, Cfg::CTAS>();
    if (st != GMG_OK) return st;
  }
  return prepare_closure_solo(DIM, K);
}

}  // namespace

int prepare_closure_f64(int dim, int k) { GMG_DISPATCH(prepare_all, dim, k) }

template <>
int upload_closure_tables<double>(int k, const double* Mp, const double* Kp, const double* That) {
  const int st = pl_upload(k, Mp, Kp, That);
  return st != GMG_OK ? st : upload_closure_solo_tables(k, Mp, Kp, That);
}

template <>
int launch_patch_table<double>(int dim, int k, const PatchLaunch* pls, double* const* us, const double* const* bs, int n,
                             const double* dinv, int ppc, cudaStream_t s) {
  GMG_DISPATCH(table_launches, dim, k, pls, us, bs, n, dinv, ppc, s)
}

template <>
int launch_patch_colour<double>(const PatchLaunch& pl, double* u, const double* b, const double* dinv, cudaStream_t s) {
  return launch_patch_table<double>(pl.g.dim, pl.g.k, &pl, &u, &b, 1, dinv, 0, s);
}

}  // namespace gmg
