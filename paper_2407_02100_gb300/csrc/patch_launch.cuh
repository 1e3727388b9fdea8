// Launchers for one scalar type; included after patch_kernels.cuh by
// patch_f64.cu / patch_f32.cu.
#pragma once
#include <algorithm>
#include <vector>

#include "../../include/gmg.h"
#include "coef_split.h"
#include "patch_dispatch.h"
#include "tma_host.h"
#include "staged_apply.cuh"

namespace gmg {
namespace GMG_NS {

constexpr int kApplyThreads = 128;

// Tile of the operator kernel (cells per direction x, y, z) and its threads.
// A tile recomputes a halo of K + 1 nodes below it in each direction, so
// flat tiles (large in x and y, one cell in z) do less redundant work; the
// shapes below were measured on GB300 (3D, against cubes): FP64 k = 3 -34 %,
// k = 4 -37 %, k = 7 -39 %; FP32 k = 3 -49 %, k = 7 -50 %; FP32 k = 4 and the
// small degrees are fastest with cubes.
template <int DIM, int K>
struct ApplyCfg {
  static constexpr bool F64 = sizeof(T) == 8;
  static constexpr int BC = DIM == 3 ? (K == 1 ? 8 : K == 2 ? 4 : K <= 4 ? 2 : 1)
                                     : (K == 1 ? 16 : K == 2 ? 8 : K <= 4 ? 4 : 2);
  static constexpr bool FLAT = DIM == 3 && (F64 ? (K >= 3 && K <= 7) : (K == 3 || K == 7));
  static constexpr int BX = !FLAT ? BC : K == 3 ? (F64 ? 8 : 4) : K == 4 ? 8 : K == 7 ? 4 : 2;
  static constexpr int BY = !FLAT ? BC : K == 3 ? (F64 ? 8 : 4) : K == 4 ? 4 : 2;
  static constexpr int BZ = FLAT ? 1 : BC;
  static constexpr int NT = FLAT && !(K == 3 && !F64) ? 256 : kApplyThreads;
};

static int sm_count() {
  static PerDevice<int> sms_dev;
  int* const sms = sms_dev.get();
  if (!sms) return 152;
  if (*sms == 0) {
    if (cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, current_device()) != cudaSuccess || *sms <= 0)
      *sms = 152;
  }
  return *sms;
}

template <typename KernelT>
// opt the kernel in to its dynamic shared memory (the 48 KB default covers
// static plus dynamic memory, so the attribute is set whatever the size)
static int prepare(KernelT kern, int smem) {
  if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
    return GMG_ERR_CUDA;
  return GMG_OK;
}

template <int DIM, int K, int BX, int BY, int BZ, int NT>
static int apply_cfg(const ApplyLaunch& al, const T* x, T* y, const T* bvec, cudaStream_t s) {
  using D = ApplyDims<DIM, K, BX, BY, BZ>;
  auto kern = apply_kernel<DIM, K, BX, BY, BZ, NT>;
  static PerDevice<bool> ready_dev;  // attribute set once per device (also keeps graph capture free of it)
  bool* const ready = ready_dev.get();
  if (!ready) return GMG_ERR_CUDA;
  if (!*ready) {
    if (prepare(kern, D::SMEM_BYTES) != GMG_OK) return GMG_ERR_CUDA;
    *ready = true;
  }
  const long long n = al.g.n;
  const long long ntile = ((n + BX - 1) / BX) * ((n + BY - 1) / BY) * (DIM == 3 ? (n + BZ - 1) / BZ : 1);
  int grid = (int)std::min<long long>(ntile, 1 << 30);
  kern<<<grid, NT, D::SMEM_BYTES, s>>>(x, y, bvec, al);
  count_launch();
  return cudaGetLastError() == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

// degrees at which the FP64 3D three-pass form beats the tile kernel
constexpr bool staged_apply_degree(int k) { return k >= 3; }

// a tile variant of the operator if its shared memory fits, else the default
template <int DIM, int K, int BX, int BY, int BZ, int NT>
static int apply_variant(const ApplyLaunch& al, const T* x, T* y, const T* bvec, cudaStream_t s) {
  if constexpr (ApplyDims<DIM, K, BX, BY, BZ>::SMEM_BYTES <= 227 * 1024) {
    return apply_cfg<DIM, K, BX, BY, BZ, NT>(al, x, y, bvec, s);
  } else {
    using Cfg = ApplyCfg<DIM, K>;
    return apply_cfg<DIM, K, Cfg::BX, Cfg::BY, Cfg::BZ, Cfg::NT>(al, x, y, bvec, s);
  }
}

template <int DIM, int K>
static int apply_impl(const ApplyLaunch& al, const T* x, T* y, const T* bvec, cudaStream_t s) {
  if constexpr (DIM == 3 && sizeof(T) == 8 && staged_apply_degree(K))
    if (al.ws) return staged_apply_impl<K>(al, x, y, bvec, s);
  if constexpr (DIM == 3 && (K == 3 || K == 4 || K == 7)) {
    constexpr int BC = ApplyCfg<DIM, K>::BC;
    switch (al.tile) {
      case 1: return apply_variant<DIM, K, BC, BC, BC, kApplyThreads>(al, x, y, bvec, s);
      case 2: return apply_variant<DIM, K, 4, 4, 1, 128>(al, x, y, bvec, s);
      case 3: return apply_variant<DIM, K, 8, 4, 1, 256>(al, x, y, bvec, s);
      default: break;
    }
  }
  if constexpr (DIM == 2) {
    // fewer tiles than SMs: a quarter of the work per tile (same results); with
    // a thread per line and cell, Q2 32^2 FP64 15 -> 5 us
    constexpr int BC = ApplyCfg<DIM, K>::BC;
    const long long t = (al.g.n + BC - 1) / BC;
    if (t * t < sm_count()) return apply_cfg<DIM, K, BC / 2, BC / 2, 1, kApplyThreads>(al, x, y, bvec, s);
  }
  using Cfg = ApplyCfg<DIM, K>;
  static_assert(ApplyDims<DIM, K, Cfg::BX, Cfg::BY, Cfg::BZ>::SMEM_BYTES <= 227 * 1024,
                "operator tile exceeds the shared memory of a CTA");
  return apply_cfg<DIM, K, Cfg::BX, Cfg::BY, Cfg::BZ, Cfg::NT>(al, x, y, bvec, s);
}

static int upload(int k, const double* Mp, const double* Kp, const double* That, const double* Mc,
                  const double* Kc) {
  if (k < 1 || k > 8) return GMG_ERR_INVALID_ARG;
  const int C = 2 * k + 1, M = 2 * k - 1;
  std::vector<T> mp(M * C), kp(M * C), tt(M * M), mc((k + 1) * (k + 1)), kc((k + 1) * (k + 1));
  for (int i = 0; i < M * C; ++i) { mp[i] = (T)Mp[i]; kp[i] = (T)Kp[i]; }
  for (int i = 0; i < M * M; ++i) tt[i] = (T)That[i];
  for (int i = 0; i < (k + 1) * (k + 1); ++i) { mc[i] = (T)Mc[i]; kc[i] = (T)Kc[i]; }
  cudaError_t e = cudaSuccess;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mp, mp.data(), mp.size() * sizeof(T), off_patch(k) * sizeof(T)) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kp, kp.data(), kp.size() * sizeof(T), off_patch(k) * sizeof(T)) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_T, tt.data(), tt.size() * sizeof(T), off_t(k) * sizeof(T)) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mc, mc.data(), mc.size() * sizeof(T), off_cell(k) * sizeof(T)) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kc, kc.data(), kc.size() * sizeof(T), off_cell(k) * sizeof(T)) : e;
  std::vector<float> thi(M * M), tlo(M * M);
  for (int i = 0; i < M * M; ++i) {
    thi[i] = (float)That[i];
    tlo[i] = (float)(That[i] - (double)thi[i]);
  }
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Thi, thi.data(), thi.size() * sizeof(float), off_t(k) * sizeof(float)) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Tlo, tlo.data(), tlo.size() * sizeof(float), off_t(k) * sizeof(float)) : e;
  std::vector<float> mhi(M * C), mlo(M * C), khi(M * C), klo(M * C);
  for (int i = 0; i < M * C; ++i) {
    mhi[i] = (float)Mp[i];
    mlo[i] = (float)(Mp[i] - (double)mhi[i]);
  }
  split_patch_stiffness(Kp, k, khi, klo);
  const size_t po = off_patch(k) * sizeof(float), pb = mhi.size() * sizeof(float);
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mphi, mhi.data(), pb, po) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mplo, mlo.data(), pb, po) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kphi, khi.data(), pb, po) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kplo, klo.data(), pb, po) : e;
  const int nc = (k + 1) * (k + 1);
  std::vector<float> mch(nc), mcl(nc), kch(nc), kcl(nc);
  for (int i = 0; i < nc; ++i) {
    mch[i] = (float)Mc[i];
    mcl[i] = (float)(Mc[i] - (double)mch[i]);
  }
  split_zero_sum_rows(Kc, k + 1, k + 1, kch, kcl);
  const size_t co = off_cell(k) * sizeof(float), cb = nc * sizeof(float);
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mchi, mch.data(), cb, co) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Mclo, mcl.data(), cb, co) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kchi, kch.data(), cb, co) : e;
  e = e == cudaSuccess ? cudaMemcpyToSymbol(c_Kclo, kcl.data(), cb, co) : e;
  return e == cudaSuccess ? GMG_OK : GMG_ERR_CUDA;
}

}  // namespace GMG_NS

template <>
int upload_patch_tables<GMG_T>(int k, const double* Mp, const double* Kp, const double* That,
                               const double* Mc, const double* Kc, cudaStream_t) {
  const int st = GMG_NS::upload(k, Mp, Kp, That, Mc, Kc);
  if (st != GMG_OK) return st;
  return upload_closure_tables<GMG_T>(k, Mp, Kp, That);
}

template <>
int launch_apply<GMG_T>(const ApplyLaunch& al, const GMG_T* x, GMG_T* y, const GMG_T* bvec,
                        cudaStream_t s) {
  GMG_DISPATCH(GMG_NS::apply_impl, al.g.dim, al.g.k, al, x, y, bvec, s)
}

}  // namespace gmg
