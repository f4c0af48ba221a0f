// Passes of the complex128 form in 64-bit fixed point (wp_fx.h): a tile is held as integers
// with one exponent through the transforms and factors of the pass. Tiles, stage plan and
// thread mapping are those of the fixed-shape kernels of wp_kernels.cuh (2048 points, 256
// threads, n = 32..2048, the lengths whose stages unroll); the passes that form observable
// sums or apply a grid potential stay in FP64.
//
// Bound by the integer pipe (64 lanes per clock; ncu on 256^3: 61 % busy over the launch,
// FP64 before 92 %) and by instruction issue (62 %). Measured on the 256^3 barrier, CUDA
// events in the step, FP64 before and fixed point now: FFT-only pass 617 -> 162 us, kinetic
// pass 1411 -> 333 us, potential pass 1118 -> 352 us.
//
// In memory a state is complex128 at the ends of a chunk of steps and in fixed point between
// its passes (F_IN_FX, F_OUT_FX): the conversions between doubles and integers are about
// 130 instructions per point and pass, those of the stored fixed-point form about 40 (FFT-only
// pass 187 -> 162 us under ncu).
//
#pragma once

#include "wp_fx.h"
#include "wp_kernels.cuh"

namespace wp {

namespace fxp {

__device__ __forceinline__ uint32_t whi(double x) { return (uint32_t)__double2hiint(x); }
__device__ __forceinline__ uint32_t wlo(double x) { return (uint32_t)__double2loint(x); }

// The high word of |v|, rounded down, from that of v.
__device__ __forceinline__ uint32_t absh(uint32_t h) { return h ^ (uint32_t)((int32_t)h >> 31); }
__device__ __forceinline__ uint32_t absh(int64_t v) { return absh((uint32_t)(v >> 32)); }

// The largest line sum of the tile (L: the thread's part of line tid mod C's) and the union
// of the threads' `any`. red, redm: 256 and 8 words, not used by anything else between the
// barriers before and after the call.
template <int LOGC>
__device__ __forceinline__ uint32_t tile_sum(uint32_t L, uint32_t& any, uint32_t* red, uint32_t* redm) {
  constexpr int C = 1 << LOGC;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int o = C; o < 32; o <<= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  any = __reduce_or_sync(0xffffffffu, any);
  constexpr int CW = C < 32 ? C : 32;  // lines a warp meets; of 64 lines odd and even warps meet one half each
  if (lane < CW) red[warp * CW + lane] = L;
  if (lane == 0) redm[warp] = any;
  __syncthreads();
  uint32_t t[2] = {0, 0};
#pragma unroll
  for (int w = 0; w < 8; w++) {
    t[C > 32 ? w & 1 : 0] += red[w * CW + (lane & (CW - 1))];
    any |= redm[w];
  }
  return __reduce_max_sync(0xffffffffu, max(t[0], t[1]));
}
// v shifted right by k (the last bit set, as fx_from_double), left for k < 0.
__device__ __forceinline__ int64_t shift_jam(int64_t v, int32_t k) {
  if (k < 0) return (int64_t)((uint64_t)v << -k);
  const uint32_t lo = fx_shr64((uint32_t)v, (uint32_t)(v >> 32), (uint32_t)k) | 1u;
  return (int64_t)(((uint64_t)(uint32_t)((int32_t)(v >> 32) >> k) << 32) | lo);
}

// One Stockham stage (stage_fixed) with its scaling.
template <int LOGN, int LOGC, int LS, int LOGNS>
__device__ __forceinline__ void stage(cx<int64_t>* s, const FxRec* __restrict__ tw, uint32_t sh, int tid) {
  constexpr int LR = wp_stage_radix_log(LOGN, LOGNS);
  constexpr int R = 1 << LR, C = 1 << LOGC, NR = 1 << (LOGN - LR), B = 8 / R, NS = 1 << LOGNS;
  cx<int64_t> v[B][R];
#pragma unroll
  for (int b = 0; b < B; b++) {
    const int bi = tid + b * 256, l = bi & (C - 1), j = bi >> LOGC;
#pragma unroll
    for (int r = 0; r < R; r++) v[b][r] = s[(j + r * NR) * LS + l];
    if (LOGNS > 0) {
      const FxRec* e = tw + (j & (NS - 1)) * (R - 1);
      v[b][0] = mk(v[b][0].re >> (2u - sh), v[b][0].im >> (2u - sh));
#pragma unroll
      for (int r = 1; r < R; r++) v[b][r] = fx_cmul(v[b][r], e[r - 1], sh);
    }
    fx_dft<R>(v[b]);
  }
  __syncthreads();
#pragma unroll
  for (int b = 0; b < B; b++) {
    const int bi = tid + b * 256, l = bi & (C - 1), j = bi >> LOGC;
    const int d0 = ((j >> LOGNS) << (LOGNS + LR)) + (j & (NS - 1));
#pragma unroll
    for (int r = 0; r < R; r++) s[(d0 + (r << LOGNS)) * LS + l] = v[b][r];
  }
  __syncthreads();
}
// The forward transform of every line of the tile. The inverse one is the same on points
// with real and imaginary parts exchanged, before and after.
template <int LOGN, int LOGC, int LS, int LOGNS = 0, int T = 0>
__device__ __forceinline__ void fft(cx<int64_t>* s, const FxRec* __restrict__ tw, const FxSchedule& sc, int tid) {
  if constexpr (LOGNS < LOGN) {
    stage<LOGN, LOGC, LS, LOGNS>(s, tw + wp_stage_tw_offset(LOGN, LOGNS), sc.at[T], tid);
    fft<LOGN, LOGC, LS, LOGNS + wp_stage_radix_log(LOGN, LOGNS), T + 1>(s, tw, sc, tid);
  }
}

// Point e of the tile, its parts exchanged when swap is 1.
__device__ __forceinline__ void put(cx<int64_t>* s, int e, int swap, int64_t re, int64_t im) {
  int64_t* q = reinterpret_cast<int64_t*>(s + e);
  q[swap] = re;
  q[1 - swap] = im;
}
__device__ __forceinline__ cx<int64_t> get(const cx<int64_t>* s, int e, int swap) {
  const int64_t* q = reinterpret_cast<const int64_t*>(s + e);
  return mk(q[swap], q[1 - swap]);
}

// The factor exp(-i theta) of a Gaussian term (FP64, as apply_gauss_phase).
__device__ __forceinline__ cx<int64_t> gauss_phase(cx<int64_t> v, double th, int& bad) {
  if (fabs(th) < 0x1p-60) return v;
  const cx<double> f = apply_gauss_phase(mk(1.0, 0.0), th);
  const FxRec w = fx_rec_of(f.re, f.im);
  bad |= w.bad;
  return fx_cmul(v, w);
}

// x 2^e at the ends of a double's range.
template <class T>
__device__ __noinline__ cx<double> scaled(cx<T> x, int e) {
  return mk(scalbn(__ll2double_rn(x.re), e), scalbn(__ll2double_rn(x.im), e));
}

// v: the thread's points i0 + k 256/C of line tid mod C (fixed_walk), loaded by the caller.
template <int LOGN, bool CONTIG>
__device__ __forceinline__ void pass(const PassParams<double>& p, cx<int64_t>* s, int64_t tile, cx<double> (&v)[8]) {
  using SH = FixShape<LOGN, CONTIG>;
  constexpr int LOGC = SH::logC, C = 1 << LOGC, LS = SH::LS, ISTEP = 256 >> LOGC;
  __shared__ uint32_t red[2][256];
  __shared__ uint32_t redm[3][8];
  __shared__ int spoil;  // a factor that is not finite spoils its tile
  const int tid = threadIdx.x, l = tid & (C - 1), i0 = tid >> LOGC;
  const uint32_t f = p.flags;
  const FxRec* tw = p.Wfx;

  int64_t o0, cb, base, es;
  int ll, ii;
  tile_origin(p, SH(), tile, o0, cb);
  fixed_walk<double, SH>(p, o0, cb, ll, ii, base, es);
  cx<double>* dst = p.out + base;
  const int64_t step = es * ISTEP;
  const bool in_fx = (f & F_IN_FX) && p.fx_state, out_fx = (f & F_OUT_FX) && p.fx_state;

  // Load: the tile's exponent (the largest leading bit), its bounds M and S, the integers.
  // An integer x of the tile stands for x 2^(ex - 1085).
  auto tile_max = [&](uint32_t m) {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((tid & 31) == 0) redm[0][tid >> 5] = m;
    if (tid == 0) spoil = 0;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; w++) m = max(m, redm[0][w]);
    return m;
  };
  // a tile that is all zero stays so; a value that is not finite spoils its tile
  auto fill = [&](bool finite) {
    const double z = finite ? 0.0 : (out_fx ? __longlong_as_double(63) : __longlong_as_double(0x7ff8000000000000ll));
#pragma unroll
    for (int k = 0; k < 8; k++) dst[k * step] = mk(z, z);
  };
  FxSchedule sc;
  int32_t ex;
  uint32_t L = 0;
  const bool ph = (f & F_PHASE) != 0, kin = (f & F_KIN) != 0;
  int swap = (f & F_IFFT) ? 1 : 0;  // whether the tile's points have their parts exchanged
  if (in_fx) {
    uint32_t m = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) m = max(m, fx_code(wlo(v[k].re), wlo(v[k].im)));
    m = tile_max(m);
    if (m == 0u || m == (uint32_t)kFxNan) return fill(m == 0u);
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t d = m - fx_code(wlo(v[k].re), wlo(v[k].im));
      const uint32_t ar = fx_shr64(absh(whi(v[k].re)), 0u, d), ai = fx_shr64(absh(whi(v[k].im)), 0u, d);
      any |= ar | ai;
      L += (ar >> 11) + (ai >> 11) + 2u;
    }
    const uint32_t Lm = tile_sum<LOGC>(L, any, red[0], redm[1]);
    sc = fx_schedule<LOGN>(65 - __clz((int)any), fx_sum_bits(Lm));
    ex = (int32_t)m - kFxBias + sc.first;
    const uint32_t right = sc.first > 0 ? (uint32_t)sc.first : 0u, left = sc.first < 0 ? (uint32_t)-sc.first : 0u;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rl = wlo(v[k].re), il = wlo(v[k].im), d = m - fx_code(rl, il) + right;
      put(s, (i0 + k * ISTEP) * LS + l, swap, (int64_t)((uint64_t)fx_align(rl, (int32_t)whi(v[k].re), d) << left),
          (int64_t)((uint64_t)fx_align(il, (int32_t)whi(v[k].im), d) << left));
    }
  } else {
    auto top = [&] {
      uint32_t m = 0;
#pragma unroll
      for (int k = 0; k < 8; k++) m = max(m, max(whi(v[k].re) & 0x7fffffffu, whi(v[k].im) & 0x7fffffffu));
      return tile_max(m);
    };
    uint32_t m = top();
    int32_t off = 0;  // the integers hold the tile times 2^-off
    if (m < (70u << 20)) {
      // all below 2^-953: lift the tile off the denormals
      __syncthreads();
      off = -900;
#pragma unroll
      for (int k = 0; k < 8; k++) v[k] = mk(v[k].re * 0x1p900, v[k].im * 0x1p900);
      m = top();
    }
    if (m == 0u || m >= 0x7ff00000u) return fill(m == 0u);
    const uint32_t E = m >> 20;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      L += fx_mag(whi(v[k].re), E - ((whi(v[k].re) >> 20) & 0x7ffu));
      L += fx_mag(whi(v[k].im), E - ((whi(v[k].im) >> 20) & 0x7ffu));
    }
    uint32_t any = 0;
    sc = fx_schedule<LOGN>(64, fx_sum_bits(tile_sum<LOGC>(L, any, red[0], redm[1])));
    const uint32_t E2 = E + (uint32_t)sc.first;
    ex = (int32_t)E2 + off;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rh = whi(v[k].re), ih = whi(v[k].im);
      put(s, (i0 + k * ISTEP) * LS + l, swap, fx_from_double(rh, wlo(v[k].re), E2 - ((rh >> 20) & 0x7ffu)),
          fx_from_double(ih, wlo(v[k].im), E2 - ((ih >> 20) & 0x7ffu)));
    }
  }
  __syncthreads();

  // Transform (inverse, or the forward one of a kinetic pass), factors, transform (forward, or
  // the inverse one of a kinetic pass): one copy of the transform's code for both, because
  // the instruction cache holds little more (two copies waited on instruction fetches).
  const bool t0 = kin || (f & F_IFFT), t1 = kin || (f & F_FFT), mid = ph || kin || (t0 && t1);
#pragma unroll 1
  for (int it = 0; it < 2; it++) {
    if (it == 0 ? t0 : t1) {
      fft<LOGN, LOGC, LS>(s, tw, sc, tid);
      ex += sc.total - sc.first;
    }
    if (it == 1 || !mid) continue;
    // the factors of the middle of the pass, and the new bound for the transform after it
    const int64_t line = CONTIG ? o0 + l : cb + l;
    LineRec<double> rec = {};
    if (ph) rec = p.lines_phase[line];
    if (kin) rec = p.lines_kin[line];
    // |L| <= 1: its exponent distance from 1 is the shift
    const uint32_t rh = whi(rec.L.w.re), ih = whi(rec.L.w.im);
    const FxRec Lr = fx_rec(fx_from_double(rh, wlo(rec.L.w.re), 1023u - ((rh >> 20) & 0x7ffu)),
                            fx_from_double(ih, wlo(rec.L.w.im), 1023u - ((ih >> 20) & 0x7ffu)));
    const bool sep = kin || (ph && p.sep);  // without additive terms the factors are exactly 1
    const FxRec* A = kin ? p.Kfx : p.Pfx;
    const bool g0 = ph && p.ngauss > 0 && gauss_line_active(rec.g[0]);
    const bool g1 = ph && p.ngauss > 1 && gauss_line_active(rec.g[1]);
    const double* G0 = p.G[0][p.axis];
    const double* G1 = p.G[1][p.axis];
    int bad = sep && (rh & 0x7ff00000u) == 0x7ff00000u;
    cx<int64_t> x[8];
    uint32_t any = 0;
    L = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int i = i0 + k * ISTEP;
      x[k] = get(s, i * LS + l, swap);
      if (sep) {
        const FxRec a = A[i];
        bad |= a.bad;
        x[k] = fx_cmul(x[k], a);
        x[k] = fx_cmul(x[k], Lr);
      }
      if (g0) x[k] = gauss_phase(x[k], rec.g[0] * G0[i], bad);
      if (g1) x[k] = gauss_phase(x[k], rec.g[1] * G1[i], bad);
      const uint32_t ar = absh(x[k].re), ai = absh(x[k].im);
      any |= ar | ai;
      L += (ar >> 11) + (ai >> 11) + 2u;
    }
    if (bad) spoil = 1;
    swap = kin ? 1 : 0;
    if (t0 && t1) {
      // the transform before has changed the bounds: a new scale
      const uint32_t Lm = tile_sum<LOGC>(L, any, red[1], redm[2]);
      sc = fx_schedule<LOGN>(65 - __clz((int)any), fx_sum_bits(Lm));
      ex += sc.first;
#pragma unroll
      for (int k = 0; k < 8; k++)
        put(s, (i0 + k * ISTEP) * LS + l, swap, shift_jam(x[k].re, sc.first), shift_jam(x[k].im, sc.first));
    } else {
#pragma unroll
      for (int k = 0; k < 8; k++) s[(i0 + k * ISTEP) * LS + l] = x[k];
    }
    __syncthreads();
  }
  if (kin) ex -= p.g.ln[0] + p.g.ln[1] + p.g.ln[2];  // 1/N
  if (out_fx) {
    // each thread's eight points shifted up together, so that the code bits cost nothing of
    // their largest
    cx<int64_t> x[8];
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      x[k] = get(s, (i0 + k * ISTEP) * LS + l, swap);
      any |= absh(x[k].re) | absh(x[k].im);
    }
    const uint32_t up = (uint32_t)max(__clz((int)any) - 1, 0);
    int32_t code = ex - (int32_t)up + kFxBias;
    if (code <= 0 || spoil) {
      code = spoil ? kFxNan : 0;
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint64_t re = (uint64_t)x[k].re << up, im = (uint64_t)x[k].im << up;
      const uint32_t rl = ((uint32_t)re & ~63u) | ((uint32_t)code >> 6), il = ((uint32_t)im & ~63u) | ((uint32_t)code & 63u);
      dst[k * step] = mk(__hiloint2double((int)(re >> 32), (int)rl), __hiloint2double((int)(im >> 32), (int)il));
    }
    return;
  }
  const bool chk = ex < 200 || ex > 1900;  // the range of a double may be left
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const cx<int64_t> x = get(s, (i0 + k * ISTEP) * LS + l, swap);
    uint32_t rh, rl, ih, il;
    fx_to_double(x.re, ex, rh, rl);
    fx_to_double(x.im, ex, ih, il);
    cx<double> y = mk(__hiloint2double((int)rh, (int)rl), __hiloint2double((int)ih, (int)il));
    if (chk) y = scaled(x, ex - 1085);
    if (spoil) y = mk(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
    dst[k * step] = y;
  }
}

template <int LOGN, bool CONTIG>
__device__ __forceinline__ void load(const cx<double>* in, int log_inner, int64_t tile, cx<double> (&v)[8]) {
  using SH = FixShape<LOGN, CONTIG>;
  constexpr int ISTEP = 256 >> SH::logC;
  const int l = threadIdx.x & ((1 << SH::logC) - 1), i0 = threadIdx.x >> SH::logC;
  int64_t base, es;
  if (CONTIG) {
    base = (((tile << SH::logC) + l) << SH::logn) + i0;
    es = 1;
  } else {
    const int tpo = log_inner - SH::logC;
    const int64_t o0 = tile >> tpo, cb = (tile & ((int64_t(1) << tpo) - 1)) << SH::logC;
    es = int64_t(1) << log_inner;
    base = (((o0 << SH::logn) + i0) << log_inner) + cb + l;
  }
  const cx<double>* q = in + base;
#pragma unroll
  for (int k = 0; k < 8; k++) v[k] = q[k * es * ISTEP];
}

template <int LOGN, bool CONTIG>
__global__ void __launch_bounds__(256, 4) k_pass_fx(const PassParams<double> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  cx<double> v[8];
  load<LOGN, CONTIG>(p.in, p.log_inner, blockIdx.x, v);
  pass<LOGN, CONTIG>(p, reinterpret_cast<cx<int64_t>*>(smem_raw), blockIdx.x, v);
}

}  // namespace fxp
}  // namespace wp
