// Patch sweep and level operator kernels in double precision.
#define GMG_T double
#define GMG_NS f64
#include "patch_kernels.cuh"
#include "patch_launch.cuh"
#include "small_kernels.cuh"

namespace gmg {
namespace f64 {

// Closure form with one patch per thread (patch_colour_kernel), 3D degrees 7
// and 8: two such patches do not fit in the shared memory of a CTA
// (pair_closure.cuh serves everything else).
template <int K, int ME>
static int line_launch(PatchTable& tab, const double* dinv, cudaStream_t s) {
  constexpr int NT = 256;
  using Z = SweepSmem<3, K, (ME > 0)>;
  constexpr int SMEM = Z::per_patch(1) * (int)sizeof(double) + (ME > 0 ? 128 : 0);
  static_assert(SMEM <= 227 * 1024, "sweep kernel shared memory exceeds the per-CTA limit");
  auto kern = patch_colour_kernel<3, K, NT, 1, 1, ME>;
  static PerDevice<int> slots_dev;  // resident CTAs (persistent grid)
  int* const slots = slots_dev.get();
  if (!slots) return GMG_ERR_CUDA;
  if (*slots == 0) {
    int per_sm = 0;
    if (prepare(kern, SMEM) != GMG_OK) return GMG_ERR_CUDA;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, NT, SMEM) != cudaSuccess || per_sm <= 0)
      return GMG_ERR_CUDA;
    *slots = per_sm * sm_count();
  }
  int groups = 0;
  for (int i = 0; i < tab.n; ++i) {
    tab.e[i].group_begin = groups;
    groups += tab.e[i].n_patches;
  }
  tab.total_groups = groups;
  if (groups <= 0) return GMG_OK;
  TmaMaps<ME> maps;
  if constexpr (ME > 0) {
    for (int i = 0; i < tab.n; ++i) {
      const PatchEntry& e = tab.e[i];
      if (!tma_encode(&maps.u[i], e.u, 8, 3, e.N, e.py, e.pz, Z::XU, Z::C) ||
          !tma_encode(&maps.b[i], e.b, 8, 3, e.N, e.py, e.pz, Z::XB, Z::M))
        return GMG_ERR_CUDA;
    }
  }
  int* const flag = device_wait_flag();
  if (!flag) return GMG_ERR_CUDA;
  kern<<<std::min(groups, *slots), NT, SMEM, s>>>(tab, dinv, maps, flag);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

template <int K>
static int line_table(const PatchLaunch* pls, double* const* us, const double* const* bs, int n, const double* dinv,
                      cudaStream_t s) {
  for (int i0 = 0; i0 < n; i0 += kMaxTable) {
    PatchTable tab;
    tab.n = 0;
    tab.mode = pls[i0].mode;
    tab.omega = pls[i0].omega;
    bool tma = true;  // else one cp.async per element
    for (int i = i0; i < std::min(n, i0 + kMaxTable); ++i) {
      if (pls[i].n_patches <= 0) continue;
      fill_entry(tab.e[tab.n], pls[i], us[i], bs[i]);
      const PatchEntry& e = tab.e[tab.n++];
      tma = tma && e.N >= 2 && tma_vector_ok(e.u, 8, 3, e.py, e.pz) && tma_vector_ok(e.b, 8, 3, e.py, e.pz);
    }
    if (tab.n == 0) continue;
    const int st = !tma ? line_launch<K, 0>(tab, dinv, s)
                 : tab.n == 1 ? line_launch<K, 1>(tab, dinv, s) : line_launch<K, kMaxTable>(tab, dinv, s);
    if (st != GMG_OK) return st;
  }
  return GMG_OK;
}

}  // namespace f64

int launch_line_table(int k, const PatchLaunch* pls, double* const* us, const double* const* bs, int n,
                      const double* dinv, cudaStream_t s) {
  return k == 7 ? f64::line_table<7>(pls, us, bs, n, dinv, s) : f64::line_table<8>(pls, us, bs, n, dinv, s);
}

bool staged_apply_preferred(int dim, int k) { return dim == 3 && f64::staged_apply_degree(k); }

}  // namespace gmg
