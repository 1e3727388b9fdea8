// Host helpers of the kernel launchers: the dispatch on dimension and degree,
// and a launch's entry in a PatchTable.
#pragma once
#include "../../include/gmg.h"
#include "kernels.h"

#define GMG_DISPATCH(FN, DIMV, KV, ...)                                  \
  switch ((DIMV) * 16 + (KV)) {                                          \
    case 2 * 16 + 1: return FN<2, 1>(__VA_ARGS__);                       \
    case 2 * 16 + 2: return FN<2, 2>(__VA_ARGS__);                       \
    case 2 * 16 + 3: return FN<2, 3>(__VA_ARGS__);                       \
    case 2 * 16 + 4: return FN<2, 4>(__VA_ARGS__);                       \
    case 2 * 16 + 5: return FN<2, 5>(__VA_ARGS__);                       \
    case 2 * 16 + 6: return FN<2, 6>(__VA_ARGS__);                       \
    case 2 * 16 + 7: return FN<2, 7>(__VA_ARGS__);                       \
    case 2 * 16 + 8: return FN<2, 8>(__VA_ARGS__);                       \
    case 3 * 16 + 1: return FN<3, 1>(__VA_ARGS__);                       \
    case 3 * 16 + 2: return FN<3, 2>(__VA_ARGS__);                       \
    case 3 * 16 + 3: return FN<3, 3>(__VA_ARGS__);                       \
    case 3 * 16 + 4: return FN<3, 4>(__VA_ARGS__);                       \
    case 3 * 16 + 5: return FN<3, 5>(__VA_ARGS__);                       \
    case 3 * 16 + 6: return FN<3, 6>(__VA_ARGS__);                       \
    case 3 * 16 + 7: return FN<3, 7>(__VA_ARGS__);                       \
    case 3 * 16 + 8: return FN<3, 8>(__VA_ARGS__);                       \
    default: return GMG_ERR_INVALID_ARG;                                 \
  }

namespace gmg {

inline void fill_entry(PatchEntry& e, const PatchLaunch& pl, void* u, const void* b) {
  e.N = pl.g.N;
  e.py = pl.g.py;
  e.pz = pl.g.pz;
  for (int a = 0; a < 3; ++a) {
    e.first[a] = pl.first[a];
    e.count[a] = pl.count[a];
  }
  e.n_patches = pl.n_patches;
  e.group_begin = 0;
  e.sb = pl.sb;
  e.u = u;
  e.b = b;
  e.plist = pl.plist;
}

}  // namespace gmg
