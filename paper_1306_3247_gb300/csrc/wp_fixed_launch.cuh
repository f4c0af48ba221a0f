// Host launchers of the fixed-size pass kernels (n = 32..2048 points per line, or 64..1024:
// kAllLengths; 2048-element tiles, 256 threads), shared by the per-precision translation units
// wp_fixed_*.cu. OBS selects the variant that also forms the observable partial sums,
// GRID the one that applies a static grid potential (contiguous passes only).
#pragma once

#include <type_traits>

#include "wp_kernels.cuh"

namespace wp {
namespace fixed_detail {

// The kernel of a shape: complex128 passes without a grid in fixed point, those with one in
// FP64 with their own register bound.
template <class T, int LOGN, bool CONTIG, bool OBS, bool GRID>
constexpr auto kernel_of() {
  if constexpr (std::is_same<T, double>::value && !OBS && !GRID)
    return &fxp::k_pass_fx<LOGN, CONTIG>;
  else if constexpr (std::is_same<T, double>::value && !GRID)
    return &fxp::k_pass_fx_obs<LOGN, CONTIG>;
  else if constexpr (std::is_same<T, double>::value)
    return &k_pass_fixed_f64<LOGN, CONTIG, OBS, GRID>;
  else
    return &k_pass_fixed<T, LOGN, CONTIG, OBS, GRID>;
}

template <class T, bool OBS, bool GRID>
constexpr bool kAllLengths = !GRID && (!OBS || std::is_same<T, double>::value);
template <class T, bool OBS, bool GRID>
constexpr int kLogMin = kAllLengths<T, OBS, GRID> ? kFixedLogMin : kFixedObsLogMin;
template <class T, bool OBS, bool GRID>
constexpr int kLogMax = kAllLengths<T, OBS, GRID> ? kFixedLogMax : kFixedObsLogMax;

template <class T, bool OBS, bool GRID, int LOGN>
cudaError_t launch_n(const PassParams<T>& p, unsigned ntiles, size_t smem, cudaStream_t st) {
  if (p.log_inner == 0) {
    launch_dep(kernel_of<T, LOGN, true, OBS, GRID>(), ntiles, 256, smem, st, p);
  } else {
    if constexpr (GRID) return cudaErrorInvalidConfiguration;
    else launch_dep(kernel_of<T, LOGN, false, OBS, false>(), ntiles, 256, smem, st, p);
  }
  return cudaGetLastError();
}

template <class T, bool OBS, bool GRID, int LOGN>
cudaError_t set_limit(int smem) {
  const cudaFuncAttribute a = cudaFuncAttributeMaxDynamicSharedMemorySize;
  cudaError_t e = cudaFuncSetAttribute(kernel_of<T, LOGN, true, OBS, GRID>(), a, smem);
  if constexpr (!GRID)
    if (e == cudaSuccess) e = cudaFuncSetAttribute(kernel_of<T, LOGN, false, OBS, false>(), a, smem);
  return e;
}

template <class T, bool OBS, bool GRID, int LOGN = kLogMin<T, OBS, GRID>>
int launch(const PassParams<T>& p, unsigned ntiles, size_t smem, void* stream) {
  if constexpr (LOGN > kLogMax<T, OBS, GRID>) {
    return (int)cudaErrorInvalidConfiguration;
  } else {
    if (p.logn != LOGN) return launch<T, OBS, GRID, LOGN + 1>(p, ntiles, smem, stream);
    return (int)launch_n<T, OBS, GRID, LOGN>(p, ntiles, smem, (cudaStream_t)stream);
  }
}

template <class T, bool OBS, bool GRID, int LOGN = kLogMin<T, OBS, GRID>>
int limit(size_t smem) {
  if constexpr (LOGN > kLogMax<T, OBS, GRID>) {
    return 0;
  } else {
    const cudaError_t e = set_limit<T, OBS, GRID, LOGN>((int)smem);
    return e == cudaSuccess ? limit<T, OBS, GRID, LOGN + 1>(smem) : (int)e;
  }
}

}  // namespace fixed_detail
}  // namespace wp

// One translation unit per (precision, variant) so that they compile in parallel.
#define WP_FIXED_TU(T, OBS, GRID, LAUNCH, LIMIT)                                            \
  namespace wp {                                                                            \
  template <>                                                                               \
  int LAUNCH<T>(const PassParams<T>& p, unsigned ntiles, size_t smem, void* stream) {       \
    return fixed_detail::launch<T, OBS, GRID>(p, ntiles, smem, stream);                     \
  }                                                                                         \
  template <>                                                                               \
  int LIMIT<T>(size_t smem) {                                                               \
    return fixed_detail::limit<T, OBS, GRID>(smem);                                         \
  }                                                                                         \
  }
