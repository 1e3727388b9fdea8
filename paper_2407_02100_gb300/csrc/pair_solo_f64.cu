// Closure form of the patch sweep in double precision, one patch per thread.
#define GMG_PAIR_ARITH SoloDF
#include "pair_closure.cuh"

namespace gmg {
namespace {

template <int DIM, int K>
int solo_launch(PatchTable& tab, const T* dinv, cudaStream_t s) {
  using Cfg = SoloCfg<DIM, K>;
  return closure_launch<DIM, K, Cfg::PP, Cfg::NT, 0>(tab, dinv, s);
}

template <int DIM, int K>
int solo_prepare() {
  using Cfg = SoloCfg<DIM, K>;
  return closure_prepare<DIM, K, Cfg::PP, Cfg::NT, 0>();
}

}  // namespace

int prepare_closure_solo(int dim, int k) { GMG_DISPATCH(solo_prepare, dim, k) }

int upload_closure_solo_tables(int k, const double* Mp, const double* Kp, const double* That) {
  return pl_upload(k, Mp, Kp, That);
}

int launch_closure_solo(int dim, int k, PatchTable& tab, const double* dinv, cudaStream_t s) {
  GMG_DISPATCH(solo_launch, dim, k, tab, dinv, s)
}

}  // namespace gmg
