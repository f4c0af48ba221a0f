// Passes over lines of 512, 1024 and 2048 points held in registers (complex64, float-float): thread t
// of a line's n/8 threads has the points t + k n/8, which are the points of its butterfly in
// the first Stockham stage and its outputs in the last one. A tile is therefore read from and
// written to global memory directly, the factors between two transforms apply in registers,
// and shared memory is crossed only between the stages of a transform: six times for two
// 1024-point transforms, against eleven with the whole tile in shared memory
// (wp_kernels.cuh), whose stages, butterflies and factors these are (an instance gives the
// same bits in a batch, which runs those).
//
// Strided axes: a block takes four (complex64) or two (float-float) adjacent columns, a
// 32-byte sector of each row; the 2048-point tiles of wp_kernels.cuh read half sectors at
// 1024 complex64 points.
//
// Bound at states that stay in L2: load latency and the shared-memory path, with 37 to 40 % of
// the warps (ncu, complex64 1024 x 1024: kinetic pass 17.0 us, potential pass 14.3; issue 36 and
// 40 %, 6 and 4 warps per issue on global loads); beyond, memory and, float-float, arithmetic.
// Measured a step against those tiles: complex64 1024 x 1024 44.8 -> 31.3 us, 512 x 512 23.4 -> 12.3, 512^3 3951 -> 3146; float-float
// 512 x 512 40.2 -> 29.0, 1024 x 1024 79.6 -> 68.4, 512^3 8569 -> 8192. At 2048 points, whose
// strided tile was one column: complex64 2048 x 1024 115 -> 51 us, float-float 193 -> 129.
#pragma once

#include "wp_kernels.cuh"

namespace wp {
namespace lp {

// WIDE (strided axes): the columns of two sectors per block.
template <class T, int LOGN, bool CONTIG, bool WIDE>
struct Shape {
  static constexpr int N = 1 << LOGN, TL = N / 8;  // threads per line
  // lines per block: 128 threads of a contiguous axis, a sector or two of columns of a strided one
  static constexpr int C = CONTIG ? (TL < 128 ? 128 / TL : 1) : (WIDE ? 64 : 32) / (int)sizeof(cx<T>);
  static constexpr int LOGC = C == 8 ? 3 : (C == 4 ? 2 : (C == 2 ? 1 : 0));
  static constexpr int NT = TL * C;
  static constexpr int LINE = N + N / 8;
  static constexpr size_t SMEM = (size_t)C * LINE * sizeof(cx<T>);
  static constexpr int MIN_BLOCKS = (sizeof(cx<T>) == 8 ? 1024 : 512) / NT;  // 64 or 128 registers
};

template <class T, int LOGN, bool CONTIG, bool WIDE>
struct Tile {
  using SH = Shape<T, LOGN, CONTIG, WIDE>;
  static constexpr int TL = SH::TL, C = SH::C;
  cx<T>* s;
  int t, l;

  // shared-memory place of point i of the thread's line, one in eight left free
  __device__ __forceinline__ cx<T>& at(int i) const {
    const int q = i + (i >> 3);
    return CONTIG ? s[l * SH::LINE + q] : s[q * C + l];
  }
  template <int LOGNS, bool INV>
  __device__ __forceinline__ void stage(cx<T> (&x)[8], const TwE<T>* __restrict__ tw) const {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), R = 1 << LR, B = 8 / R, NS = 1 << LOGNS;
    constexpr bool last = LOGNS + LR == LOGN;
    if constexpr (LOGNS > 0) {
#pragma unroll
      for (int b = 0; b < B; b++)
#pragma unroll
        for (int r = 0; r < R; r++) x[b + B * r] = at(t + b * TL + r * (SH::N / R));
    }
#pragma unroll
    for (int b = 0; b < B; b++) {
      cx<T> v[R];
#pragma unroll
      for (int r = 0; r < R; r++) v[r] = x[b + B * r];
      if constexpr (LOGNS > 0) {
        const TwE<T>* e = tw + wp_stage_tw_offset(LOGN, LOGNS) + ((t + b * TL) & (NS - 1));
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = tw_apply<INV>(v[r], e[(r - 1) * NS]);
      }
      Dft<T, R, INV>::run(v);
#pragma unroll
      for (int r = 0; r < R; r++) x[b + B * r] = v[r];
    }
    if constexpr (!last) {
      __syncthreads();  // the reads of the stage (or transform) before are done
#pragma unroll
      for (int b = 0; b < B; b++) {
        const int j = t + b * TL;
        const int d0 = ((j >> LOGNS) << (LOGNS + LR)) + (j & (NS - 1));
#pragma unroll
        for (int r = 0; r < R; r++) at(d0 + (r << LOGNS)) = x[b + B * r];
      }
      __syncthreads();
      stage<LOGNS + LR, INV>(x, tw);
    }
  }
};

// NG, SEP: Gaussian and additive terms of the potential (contiguous axis); KIN: kinetic round
// trip (strided axis).
template <class T, int LOGN, bool CONTIG, bool WIDE, int NG, bool SEP, bool KIN>
__global__ void __launch_bounds__(Shape<T, LOGN, CONTIG, WIDE>::NT, Shape<T, LOGN, CONTIG, WIDE>::MIN_BLOCKS)
    k_line_pass(const PassParams<T> p) {
  using SH = Shape<T, LOGN, CONTIG, WIDE>;
  constexpr int TL = SH::TL;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  Tile<T, LOGN, CONTIG, WIDE> tile{reinterpret_cast<cx<T>*>(smem_raw), 0, 0};
  int64_t base, es, line;
  if constexpr (CONTIG) {
    tile.t = threadIdx.x & (TL - 1);
    tile.l = threadIdx.x / TL;
    line = blockIdx.x * (int64_t)SH::C + tile.l;
    base = (line << LOGN) + tile.t;
    es = 1;
  } else {
    tile.l = threadIdx.x & (SH::C - 1);
    tile.t = threadIdx.x >> SH::LOGC;
    const int tpo = p.log_inner - SH::LOGC;
    const int64_t o = blockIdx.x >> tpo;
    line = ((blockIdx.x & ((int64_t(1) << tpo) - 1)) << SH::LOGC) + tile.l;  // column
    es = int64_t(1) << p.log_inner;
    base = (((o << LOGN) + tile.t) << p.log_inner) + line;
  }
  const int64_t step = es * TL;
  const TwE<T>* tw = reinterpret_cast<const TwE<T>*>(p.Wln);
  const cx<T>* in = p.in + base;
  cx<T> x[8];
#pragma unroll
  for (int k = 0; k < 8; k++) x[k] = in[k * step];
  const uint32_t f = p.flags;
  if constexpr (CONTIG) {
    if (f & F_IFFT) tile.template stage<0, true>(x, tw);
    if (f & F_PHASE) {
      const LineRec<T> rec = p.lines_phase[line];
      const T* G0 = p.G[0][p.axis];
      const T* G1 = p.G[1][p.axis];
      const bool g0 = NG > 0 && gauss_line_active(rec.g[0]), g1 = NG > 1 && gauss_line_active(rec.g[1]);
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const int i = tile.t + k * TL;
        if constexpr (SEP) x[k] = apply_factor_rec(x[k], p.Prec[i], rec.L);
        if constexpr (NG > 0)
          if (g0) x[k] = apply_gauss_phase(x[k], rec.g[0] * G0[i]);
        if constexpr (NG > 1)
          if (g1) x[k] = apply_gauss_phase(x[k], rec.g[1] * G1[i]);
      }
    }
    if (f & F_FFT) tile.template stage<0, false>(x, tw);
  } else if constexpr (KIN) {
    const TwE<T> L = p.lines_kin[line].L;
    tile.template stage<0, false>(x, tw);
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = apply_factor_rec(x[k], p.Krec[tile.t + k * TL], L);
    tile.template stage<0, true>(x, tw);
  } else if (f & F_IFFT) {
    tile.template stage<0, true>(x, tw);
  } else {
    tile.template stage<0, false>(x, tw);
  }
  cx<T>* out = p.out + base;
#pragma unroll
  for (int k = 0; k < 8; k++) out[k * step] = x[k];
}

// Passes these kernels serve: 512 to 2048 points under the fixed schedule, no sums, no grid
// potential, whole tiles.
template <class T>
bool applies(const PassParams<T>& p) {
  if (!p.fixed || !p.Wln || p.logn < 9 || p.logn > 11) return false;
  const uint32_t f = p.flags;
  if (f & (F_OBS_POS | F_OBS_MOM | F_NO_STORE | F_AUTOCORR)) return false;
  if (p.grid_rec && (f & F_PHASE)) return false;
  int lntot = 0;
  for (int d = 0; d < p.g.ndim; d++) lntot += p.g.ln[d];
  if (p.log_inner == 0) return !(f & F_KIN) && lntot - p.logn >= 1;
  return !(f & F_PHASE) && p.log_inner >= 2;
}

template <class T, int LOGN, bool CONTIG, bool WIDE, int NG, bool SEP, bool KIN>
cudaError_t go(const PassParams<T>& p, cudaStream_t st) {
  using SH = Shape<T, LOGN, CONTIG, WIDE>;
  auto kern = k_line_pass<T, LOGN, CONTIG, WIDE, NG, SEP, KIN>;
  static std::once_flag once;
  static cudaError_t attr = cudaSuccess;
  std::call_once(once, [&] {
    attr = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)SH::SMEM);
  });
  if (attr != cudaSuccess) return attr;
  int lntot = 0;
  for (int d = 0; d < p.g.ndim; d++) lntot += p.g.ln[d];
  const unsigned blocks = (unsigned)((int64_t(1) << (lntot - LOGN)) / SH::C);
  launch_dep(kern, blocks, SH::NT, SH::SMEM, st, p);
  return cudaGetLastError();
}

template <class T, int LOGN>
cudaError_t launch_n(const PassParams<T>& p, cudaStream_t st) {
  if (p.log_inner > 0) {
    int lntot = 0;
    for (int d = 0; d < p.g.ndim; d++) lntot += p.g.ln[d];
    const bool kin = (p.flags & F_KIN) != 0;
    // Two sectors a row once the state is beyond L2's half (64 MB), where DRAM gives single
    // sectors at a lower rate: the float-float kinetic pass of 512^3 takes 3708 us with one
    // sector and 2623 with two. Below, smaller blocks fill the chip better.
    if constexpr (LOGN <= 10)
      if (p.log_inner >= 3 && (sizeof(cx<T>) << lntot) > ((size_t)64 << 20))
        return kin ? go<T, LOGN, false, true, 0, false, true>(p, st) : go<T, LOGN, false, true, 0, false, false>(p, st);
    return kin ? go<T, LOGN, false, false, 0, false, true>(p, st) : go<T, LOGN, false, false, 0, false, false>(p, st);
  }
  const int ng = p.flags & F_PHASE ? p.ngauss : 0;
  const bool sep = (p.flags & F_PHASE) && p.sep;
  if (ng >= 2) return sep ? go<T, LOGN, true, false, 2, true, false>(p, st) : go<T, LOGN, true, false, 2, false, false>(p, st);
  if (ng == 1) return sep ? go<T, LOGN, true, false, 1, true, false>(p, st) : go<T, LOGN, true, false, 1, false, false>(p, st);
  return sep ? go<T, LOGN, true, false, 0, true, false>(p, st) : go<T, LOGN, true, false, 0, false, false>(p, st);
}

}  // namespace lp
}  // namespace wp

#define WP_LINEPASS_TU(T)                                                                        \
  namespace wp {                                                                                 \
  template <>                                                                                    \
  bool line_pass_applies<T>(const PassParams<T>& p) {                                            \
    return lp::applies<T>(p);                                                                    \
  }                                                                                              \
  template <>                                                                                    \
  int launch_line_pass<T>(const PassParams<T>& p, void* stream) {                                \
    cudaStream_t st = (cudaStream_t)stream;                                                      \
    return (int)(p.logn == 9    ? lp::launch_n<T, 9>(p, st)                                      \
                 : p.logn == 10 ? lp::launch_n<T, 10>(p, st)                                     \
                                : lp::launch_n<T, 11>(p, st));                                   \
  }                                                                                              \
  }
