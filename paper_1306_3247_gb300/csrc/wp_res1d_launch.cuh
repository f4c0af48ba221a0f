// Host launchers of the resident lines of compile-time length (n = 2^8 .. 2^14, wp_line.cuh),
// shared by the per-precision translation units wp_res1d_*.cu.
#pragma once

#include "wp_line.cuh"

namespace wp {
namespace res1d_detail {

// 16-byte elements: lines of at most 2^13 points (the longest a handle accepts)
template <class T, int LOGN>
constexpr bool supported() {
  return sizeof(cx<T>) == 8 || LOGN <= 13;
}

// Blocks (log2) of the cluster that holds a line, alone and as one of a batch. Alone, a line
// takes eight SMs (the portable cluster) as soon as each block has two warps of points:
// complex128 at 4096 points 27.8 us per step on one block, 11.0 on eight. At 1024 points one
// warp per block would be left, with nothing gained over four warps of one block. In a batch
// the lines fill the GPU by themselves and a cluster only adds exchanges (256 lines of the
// uneven batch beside its 2-D passes: 2.07 ms per 20 steps with clusters of four and eight
// for 2048 points and more, 1.66 without), so that only lines of more points than 512
// threads hold are split.
template <int LOGN>
constexpr int cluster_log() {
  return LOGN <= 10 ? 0 : (LOGN == 11 ? 2 : 3);
}
template <int LOGN>
constexpr int batch_cluster_log() {
  return LOGN <= 12 ? 0 : LOGN - 12;
}

// DEP: the kernel begins with pass_begin.
template <class SH, bool DEP, class K, class... A>
cudaError_t go(K kern, unsigned nlines, cudaStream_t st, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nlines * SH::R);
  cfg.blockDim = dim3(SH::NT + SH::TW);
  cfg.dynamicSmemBytes = SH::SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2] = {};
  unsigned n = 0;
  if (DEP) {
    at[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[n++].val.programmaticStreamSerializationAllowed = 1;
  }
  if (SH::R > 1) {
    at[n].id = cudaLaunchAttributeClusterDimension;
    at[n].val.clusterDim.x = SH::R;
    at[n].val.clusterDim.y = at[n].val.clusterDim.z = 1;
    n++;
  }
  cfg.attrs = at;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

template <class T, int LOGN>
cudaError_t launch_n(const Res1dParams<T>& p, cudaStream_t st) {
  if constexpr (supported<T, LOGN>()) {
    constexpr int LOGR = cluster_log<LOGN>();
    using SH = line::Shape<T, LOGN, LOGR>;
    return go<SH, true>(line::k_line<T, LOGN, LOGR>, 1, st, p);
  }
  return cudaErrorInvalidConfiguration;
}

template <class T, int LOGN>
cudaError_t launch_batch_n(const Res1dParams<T>* params, int ninst, int64_t nsteps, cudaStream_t st) {
  if constexpr (supported<T, LOGN>()) {
    constexpr int LOGR = batch_cluster_log<LOGN>();
    using SH = line::Shape<T, LOGN, LOGR, true>;
    return go<SH, false>(line::k_line_batch<T, LOGN, LOGR>, (unsigned)ninst, st, params, nsteps);
  }
  return cudaErrorInvalidConfiguration;
}

template <class T, int LOGN>
cudaError_t set_limit() {
  if constexpr (supported<T, LOGN>()) {
    constexpr int LOGR = cluster_log<LOGN>(), LOGB = batch_cluster_log<LOGN>();
    const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t e = cudaFuncSetAttribute(line::k_line<T, LOGN, LOGR>, a, (int)line::Shape<T, LOGN, LOGR>::SMEM);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(line::k_line_batch<T, LOGN, LOGB>, a, (int)line::Shape<T, LOGN, LOGB, true>::SMEM);
    return e;
  }
  return cudaSuccess;
}

// Calls F<LOGN>() for LOGN = logn in kRes1dLogMin .. kRes1dLogMax.
template <class F>
bool dispatch(int logn, F&& f) {
  switch (logn) {
    case 8:
      f(std::integral_constant<int, 8>());
      return true;
    case 9:
      f(std::integral_constant<int, 9>());
      return true;
    case 10:
      f(std::integral_constant<int, 10>());
      return true;
    case 11:
      f(std::integral_constant<int, 11>());
      return true;
    case 12:
      f(std::integral_constant<int, 12>());
      return true;
    case 13:
      f(std::integral_constant<int, 13>());
      return true;
    case 14:
      f(std::integral_constant<int, 14>());
      return true;
    default:
      return false;
  }
}

}  // namespace res1d_detail
}  // namespace wp

#define WP_RES1D_TU(T)                                                                                 \
  namespace wp {                                                                                       \
  template <>                                                                                          \
  int launch_res1d_fixed<T>(const Res1dParams<T>& p, void* stream) {                                   \
    cudaError_t e = cudaErrorInvalidConfiguration;                                                     \
    res1d_detail::dispatch(p.logn, [&](auto L) {                                                       \
      e = res1d_detail::launch_n<T, decltype(L)::value>(p, (cudaStream_t)stream);                      \
    });                                                                                                \
    return e == cudaSuccess ? 0 : (int)e;                                                              \
  }                                                                                                    \
  template <>                                                                                          \
  int launch_res1d_fixed_batch<T>(const Res1dParams<T>* params, int ninst, int logn, int64_t nsteps,  \
                                  void* stream) {                                                      \
    if (ninst <= 0) return 0;                                                                          \
    cudaError_t e = cudaErrorInvalidConfiguration;                                                     \
    res1d_detail::dispatch(logn, [&](auto L) {                                                         \
      e = res1d_detail::launch_batch_n<T, decltype(L)::value>(params, ninst, nsteps,                   \
                                                              (cudaStream_t)stream);                   \
    });                                                                                                \
    return e == cudaSuccess ? 0 : (int)e;                                                              \
  }                                                                                                    \
  template <>                                                                                          \
  int res1d_fixed_smem_limit_set<T>() {                                                                \
    cudaError_t e = cudaSuccess;                                                                       \
    for (int l = kRes1dLogMin; l <= kRes1dLogMax && e == cudaSuccess; l++)                             \
      res1d_detail::dispatch(l, [&](auto L) { e = res1d_detail::set_limit<T, decltype(L)::value>(); }); \
    return e == cudaSuccess ? 0 : (int)e;                                                              \
  }                                                                                                    \
  }
