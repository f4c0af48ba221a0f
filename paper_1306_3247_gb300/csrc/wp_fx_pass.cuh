// Passes of the complex128 form in 64-bit fixed point (wp_fx.h): a tile is held as integers
// with one exponent through the transforms and factors of the pass. Tiles and stage plan are
// those of the fixed-shape kernels of wp_kernels.cuh (2048 points, 256
// threads, n = 32..2048, the lengths whose stages unroll); those that form observable sums
// add them up in FP64 from the results; passes that apply a grid potential stay in FP64.
//
// Bound by the integer pipe (64 lanes per clock; ncu on 256^3: 63-69 % busy, FP64 before
// 92 %) and by instruction issue. Measured on the 256^3 barrier, CUDA events in the step, FP64
// before, fixed point with the whole tile in shared memory, and these: FFT-only pass 617, 162,
// 159 us; kinetic pass 1411, 333, 322; potential pass 1118, 352, 290. The FP64 pipe bounds the
// sums of a record (86 % busy in the position sums, 489 us).
//
// In memory a state is complex128 at the ends of a chunk of steps and in fixed point between
// its passes (F_IN_FX, F_OUT_FX): the conversions between doubles and integers are about
// 130 instructions per point and pass, those of the stored fixed-point form about 40 (FFT-only
// pass 187 -> 162 us under ncu).
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

// A tile's lines in registers and shared memory: thread t of a line's n/8 threads holds the
// points t + k n/8, which are the inputs of its butterfly in the first Stockham stage and its
// outputs in the last; shared memory is crossed between the stages of a transform only, and
// one in eight of its places is left free against bank conflicts. Contiguous axes: a line's
// threads side by side (whole sectors, and for n <= 256 a line within a warp, which then needs
// no block barrier between stages); strided axes: the tile's lines, adjacent columns, side by
// side.
template <int LOGN, bool CONTIG>
struct Tile {
  static constexpr int N = 1 << LOGN, LOGTL = LOGN - 3, TL = 1 << LOGTL, LOGC = 11 - LOGN, C = 1 << LOGC;
  static constexpr int LINE = N + N / 8;
  static_assert(C * LINE * sizeof(cx<int64_t>) == kFxTileBytes, "");
  cx<int64_t>* s;
  int t, l;
  __device__ __forceinline__ explicit Tile(void* smem)
      : s(reinterpret_cast<cx<int64_t>*>(smem)),
        t(CONTIG ? threadIdx.x & (TL - 1) : threadIdx.x >> LOGC),
        l(CONTIG ? threadIdx.x >> LOGTL : threadIdx.x & (C - 1)) {}
  // offset of the thread's point 0, and the distance of the next
  __device__ __forceinline__ int64_t base(int log_inner, int64_t tile, int64_t& step) const {
    if (CONTIG) {
      step = TL;
      return (((tile << LOGC) + l) << LOGN) + t;
    }
    const int tpo = log_inner - LOGC;
    const int64_t o0 = tile >> tpo, cb = (tile & ((int64_t(1) << tpo) - 1)) << LOGC;
    step = int64_t(TL) << log_inner;
    return (((o0 << LOGN) + t) << log_inner) + cb + l;
  }
  // index of the thread's line in the pass's line records
  __device__ __forceinline__ int64_t line(int log_inner, int64_t tile) const {
    if (CONTIG) return (tile << LOGC) + l;
    return ((tile & ((int64_t(1) << (log_inner - LOGC)) - 1)) << LOGC) + l;
  }
  __device__ __forceinline__ cx<int64_t>& at(int i) const {
    const int q = i + (i >> 3);
    return CONTIG ? s[l * LINE + q] : s[q * C + l];
  }
  __device__ __forceinline__ static void sync() {
    if constexpr (CONTIG && TL <= 32)
      __syncwarp();
    else
      __syncthreads();
  }

  // The largest line sum of the tile (L: the thread's part of its line's) and the union of
  // the threads' `any`. red, redm: 256 and 8 words, not used by anything else between the
  // barriers before and after the call.
  __device__ __forceinline__ uint32_t sum(uint32_t L, uint32_t& any, uint32_t* red, uint32_t* redm) const {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    any = __reduce_or_sync(0xffffffffu, any);
    if (lane == 0) redm[warp] = any;
    uint32_t r = 0;
    if constexpr (CONTIG) {
#pragma unroll
      for (int o = 1; o < (TL < 32 ? TL : 32); o <<= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
      if constexpr (TL < 32) L = __reduce_max_sync(0xffffffffu, L);
      if (lane == 0) red[warp] = L;
      __syncthreads();
      constexpr int WL = TL < 32 ? 1 : TL / 32;  // warps of a line
#pragma unroll
      for (int w = 0; w < 8; w += WL) {
        uint32_t u = 0;
#pragma unroll
        for (int k = 0; k < WL; k++) u += red[w + k];
        r = max(r, u);
      }
    } else {
      constexpr int CW = C < 32 ? C : 32;  // lines a warp meets; of 64 lines odd and even warps meet one half each
#pragma unroll
      for (int o = C; o < 32; o <<= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
      if (lane < CW) red[warp * CW + lane] = L;
      __syncthreads();
      uint32_t u[2] = {0, 0};
#pragma unroll
      for (int w = 0; w < 8; w++) u[C > 32 ? w & 1 : 0] += red[w * CW + (lane & (CW - 1))];
      r = __reduce_max_sync(0xffffffffu, max(u[0], u[1]));
    }
#pragma unroll
    for (int w = 0; w < 8; w++) any |= redm[w];
    return r;
  }

  // The forward transform of the tile's lines, with the scaling of sc. The inverse one is the
  // same on points with real and imaginary parts exchanged, before and after.
  template <int LOGNS = 0, int S = 0>
  __device__ __forceinline__ void fft(cx<int64_t> (&x)[8], const FxRec* __restrict__ tw, const FxSchedule& sc) const {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), R = 1 << LR, B = 8 / R, NS = 1 << LOGNS;
    if constexpr (LOGNS > 0) {
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = at(t + k * TL);
    }
#pragma unroll
    for (int b = 0; b < B; b++) {
      cx<int64_t> v[R];
#pragma unroll
      for (int r = 0; r < R; r++) v[r] = x[b + B * r];
      if constexpr (LOGNS > 0) {
        const uint32_t sh = sc.at[S];
        const FxRec* e = tw + wp_stage_tw_offset(LOGN, LOGNS) + ((t + b * TL) & (NS - 1));
        v[0] = mk(v[0].re >> (2u - sh), v[0].im >> (2u - sh));
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = fx_cmul(v[r], e[(r - 1) * NS], sh);
      }
      fx_dft<R>(v);
#pragma unroll
      for (int r = 0; r < R; r++) x[b + B * r] = v[r];
    }
    if constexpr (LOGNS + LR < LOGN) {
      sync();  // the reads of the stage (or transform) before are done
#pragma unroll
      for (int b = 0; b < B; b++) {
        const int j = t + b * TL;
        const int d0 = ((j >> LOGNS) << (LOGNS + LR)) + (j & (NS - 1));
#pragma unroll
        for (int r = 0; r < R; r++) at(d0 + (r << LOGNS)) = x[b + B * r];
      }
      sync();
      fft<LOGNS + LR, S + 1>(x, tw, sc);
    }
  }
};

// v shifted right by k (the last bit set, as fx_from_double), left for k < 0.
__device__ __forceinline__ int64_t shift_jam(int64_t v, int32_t k) {
  if (k < 0) return (int64_t)((uint64_t)v << -k);
  const uint32_t lo = fx_shr64((uint32_t)v, (uint32_t)(v >> 32), (uint32_t)k) | 1u;
  return (int64_t)(((uint64_t)(uint32_t)((int32_t)(v >> 32) >> k) << 32) | lo);
}

__device__ __forceinline__ void exchange(cx<int64_t> (&x)[8]) {
#pragma unroll
  for (int k = 0; k < 8; k++) x[k] = mk(x[k].im, x[k].re);
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

// The Gaussian terms of the thread's points in shared memory, one point at a time: the
// sine's code and registers once, and none of the pass's registers live across it.
template <class TI>
__device__ __noinline__ int gauss_points(TI ti, double a0, double a1, const double* G0, const double* G1) {
  int bad = 0;
#pragma unroll 1
  for (int k = 0; k < 8; k++) {
    const int i = ti.t + k * TI::TL;
    cx<int64_t> y = ti.at(i);
    if (gauss_line_active(a0)) y = gauss_phase(y, a0 * G0[i], bad);
    if (gauss_line_active(a1)) y = gauss_phase(y, a1 * G1[i], bad);
    ti.at(i) = y;
  }
  return bad;
}

// v: the thread's points, loaded by the caller. OBS: v returns the pass's results as doubles
// for the sums, unless the tile is empty or not finite: then its row of the sums is written
// here and the result is false.
template <int LOGN, bool CONTIG, bool OBS>
__device__ __forceinline__ bool pass(const PassParams<double>& p, void* smem, int64_t tile, cx<double> (&v)[8]) {
  using TI = Tile<LOGN, CONTIG>;
  constexpr int TL = TI::TL;
  __shared__ uint32_t red[2][256];
  __shared__ uint32_t redm[3][8];
  const TI ti(smem);
  const int tid = threadIdx.x;
  const uint32_t f = p.flags;
  const FxRec* tw = reinterpret_cast<const FxRec*>(p.Wln);
  int64_t step;
  cx<double>* dst = p.out + ti.base(p.log_inner, tile, step);
  const bool in_fx = (f & F_IN_FX) && p.fx_state, out_fx = (f & F_OUT_FX) && p.fx_state;

  // Load: the tile's exponent (the largest leading bit), its bounds M and S, the integers.
  // An integer x of the tile stands for x 2^(ex - 1085).
  auto tile_max = [&](uint32_t m) {
    m = __reduce_max_sync(0xffffffffu, m);
    if ((tid & 31) == 0) redm[0][tid >> 5] = m;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < 8; w++) m = max(m, redm[0][w]);
    return m;
  };
  // a tile that is all zero stays so; a value that is not finite spoils its tile
  auto fill = [&](bool finite) {
    const double z = finite ? 0.0 : (out_fx ? __longlong_as_double(63) : __longlong_as_double(0x7ff8000000000000ll));
#pragma unroll
    for (int k = 0; k < 8; k++)
      if (!OBS || !(f & F_NO_STORE)) dst[k * step] = mk(z, z);
    if (OBS && tid < NQ) p.partials[tile * NQ + tid] = z;
    return false;
  };
  FxSchedule sc;
  int32_t ex;
  uint32_t L = 0;
  const bool ph = CONTIG && (f & F_PHASE), kin = !CONTIG && (f & F_KIN);
  bool swap = (f & F_IFFT) != 0;  // whether the points have their parts exchanged
  cx<int64_t> x[8];
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
      L += fx_mag_int<kFxPassSum>(ar) + fx_mag_int<kFxPassSum>(ai);
    }
    const uint32_t Lm = ti.sum(L, any, red[0], redm[1]);
    sc = fx_schedule<LOGN>(65 - __clz((int)any), fx_sum_bits<kFxPassSum>(Lm));
    ex = (int32_t)m - kFxBias + sc.first;
    const uint32_t right = sc.first > 0 ? (uint32_t)sc.first : 0u, left = sc.first < 0 ? (uint32_t)-sc.first : 0u;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rl = wlo(v[k].re), il = wlo(v[k].im), d = m - fx_code(rl, il) + right;
      x[k] = mk((int64_t)((uint64_t)fx_align(rl, (int32_t)whi(v[k].re), d) << left),
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
      L += fx_mag<kFxPassSum>(whi(v[k].re), E - ((whi(v[k].re) >> 20) & 0x7ffu));
      L += fx_mag<kFxPassSum>(whi(v[k].im), E - ((whi(v[k].im) >> 20) & 0x7ffu));
    }
    uint32_t any = 0;
    sc = fx_schedule<LOGN>(64, fx_sum_bits<kFxPassSum>(ti.sum(L, any, red[0], redm[1])));
    const uint32_t E2 = E + (uint32_t)sc.first;
    ex = (int32_t)E2 + off;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rh = whi(v[k].re), ih = whi(v[k].im);
      x[k] = mk(fx_from_double(rh, wlo(v[k].re), E2 - ((rh >> 20) & 0x7ffu)),
                fx_from_double(ih, wlo(v[k].im), E2 - ((ih >> 20) & 0x7ffu)));
    }
  }
  if (swap) exchange(x);

  // Transform (inverse, or the forward one of a kinetic pass), factors, transform (forward, or
  // the inverse one of a kinetic pass): one copy of the transform's code for both, because
  // the instruction cache holds little more (two copies waited on instruction fetches).
  int spoil = 0;  // a factor that is not finite spoils its tile
  const bool t0 = kin || (f & F_IFFT), t1 = kin || (f & F_FFT), mid = ph || kin || (t0 && t1);
#pragma unroll 1
  for (int it = 0; it < 2; it++) {
    if (it == 0 ? t0 : t1) {
      ti.fft(x, tw, sc);
      ex += sc.total - sc.first;
    }
    if (it == 1 || !mid) continue;
    // the factors of the middle of the pass, and the new bound for the transform after it
    if (swap) exchange(x);
    const int64_t line = ti.line(p.log_inner, tile);
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
    if (sep) {
#pragma unroll
      for (int k = 0; k < 8; k++) {
        const FxRec a = A[ti.t + k * TL];
        bad |= a.bad;
        x[k] = fx_cmul(x[k], a);
        x[k] = fx_cmul(x[k], Lr);
      }
    }
    if (ph && p.ngauss > 0) {
      ti.sync();
#pragma unroll
      for (int k = 0; k < 8; k++) ti.at(ti.t + k * TL) = x[k];
      bad |= gauss_points(ti, g0 ? rec.g[0] : 0.0, g1 ? rec.g[1] : 0.0, G0, G1);
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = ti.at(ti.t + k * TL);
    }
    uint32_t any = 0;
    L = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t ar = absh(x[k].re), ai = absh(x[k].im);
      any |= ar | ai;
      L += fx_mag_int<kFxPassSum>(ar) + fx_mag_int<kFxPassSum>(ai);
    }
    if (t0 && t1) {
      // the transform before has changed the bounds: a new scale
      const uint32_t Lm = ti.sum(L, any, red[1], redm[2]);
      sc = fx_schedule<LOGN>(65 - __clz((int)any), fx_sum_bits<kFxPassSum>(Lm));
      ex += sc.first;
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = mk(shift_jam(x[k].re, sc.first), shift_jam(x[k].im, sc.first));
    }
    if (ph || kin) spoil = __syncthreads_or(bad);
    swap = kin;
    if (swap) exchange(x);
  }
  if (swap) exchange(x);
  if (kin) ex -= p.g.ln[0] + p.g.ln[1] + p.g.ln[2];  // 1/N
  if (!OBS && out_fx) {
    // each thread's eight points shifted up together, so that the code bits cost nothing of
    // their largest
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) any |= absh(x[k].re) | absh(x[k].im);
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
    return true;
  }
  const bool chk = ex < 200 || ex > 1900;  // the range of a double may be left
#pragma unroll
  for (int k = 0; k < 8; k++) {
    uint32_t rh, rl, ih, il;
    fx_to_double(x[k].re, ex, rh, rl);
    fx_to_double(x[k].im, ex, ih, il);
    cx<double> y = mk(__hiloint2double((int)rh, (int)rl), __hiloint2double((int)ih, (int)il));
    if (chk) y = scaled(x[k], ex - 1085);
    if (spoil) y = mk(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
    if (!OBS || !(f & F_NO_STORE)) dst[k * step] = y;
    if (OBS) v[k] = y;
  }
  return true;
}

// The tile's row of the observable sums (obs_line_row's line sums), from the thread's points
// v: position sums on a contiguous axis, momentum sums on a strided one. Every FP64
// instruction counts (one per 19 clocks and SM): the threads' eight sums cross shared memory
// once, and each warp adds up one of the eight, 8 + log2(32 / C) additions against the 40
// of a shuffle tree over all eight.
template <int LOGN, bool CONTIG>
__device__ __forceinline__ void obs_sums(const PassParams<double>& p, void* smem, int64_t tile, const cx<double> (&v)[8]) {
  using TI = Tile<LOGN, CONTIG>;
  constexpr int C = TI::C, CW = C < 32 ? C : 32;
  __shared__ double red[C][NQ];
  const TI ti(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  double q[8];
#pragma unroll
  for (int j = 0; j < 8; j++) q[j] = 0.0;
  if constexpr (CONTIG) {
    const double* G0 = p.G[0][p.axis];
    const double* G1 = p.G[1][p.axis];
    int64_t step;
    const int64_t base = ti.base(p.log_inner, tile, step);
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int i = ti.t + k * TI::TL;
      const double rho = norm2(v[k]);
      const cx<double> xx = p.Ox[i];
      q[0] += rho;
      q[1] = madd(xx.re, rho, q[1]);
      q[2] = madd(xx.im, rho, q[2]);
      q[3] = madd(p.AT[i], rho, q[3]);
      if (p.ngauss > 0) q[4] = madd(G0[i], rho, q[4]);
      if (p.ngauss > 1) q[5] = madd(G1[i], rho, q[5]);
      if (p.flags & F_AUTOCORR) {
        const cx<double> c = cmulc(v[k], p.psi0[base + k * step]);
        q[6] += c.re;
        q[7] += c.im;
      }
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const double rho = norm2(v[k]);
      const cx<double> kk = p.Ok[ti.t + k * TI::TL];
      q[0] += rho;
      q[1] = madd(kk.re, rho, q[1]);
      q[2] = madd(kk.im, rho, q[2]);
    }
  }
  constexpr int ROW = 256 + 16;  // one place in 16 left free against bank conflicts
  double* sc = reinterpret_cast<double*>(smem);
  const int e = ti.t * C + ti.l;
  __syncthreads();  // the tile is free now
#pragma unroll
  for (int j = 0; j < 8; j++) sc[j * ROW + e + (e >> 4)] = q[j];
  __syncthreads();
  double a[2] = {0.0, 0.0};
#pragma unroll
  for (int m = 0; m < 8; m++) {
    const int r = lane + 32 * m;
    a[C > 32 ? m & 1 : 0] += sc[warp * ROW + r + (r >> 4)];
  }
#pragma unroll
  for (int o = C; o < 32; o <<= 1) a[0] += __shfl_xor_sync(0xffffffffu, a[0], o);
  if (lane < CW) {
    red[lane][warp] = a[0];
    if (C > 32) red[(lane + 32) & (C - 1)][warp] = a[1];
  }
  __syncthreads();
  double lt[8];
  if (tid < C) {
#pragma unroll
    for (int j = 0; j < 8; j++) lt[j] = red[tid][j];
    int gi[3];
    const int tpo = p.log_inner - TI::LOGC;
    if (CONTIG)
      grid_index(p.g, p.axis, (tile << TI::LOGC) + tid, 0, 0, gi);
    else
      grid_index(p.g, p.axis, tile >> tpo, ((tile & ((int64_t(1) << tpo) - 1)) << TI::LOGC) + tid, 0, gi);
    obs_line_row(p, lt, gi, red[tid]);
  }
  __syncthreads();
  if (tid < NQ) {
    double sum = 0.0;
#pragma unroll 8
    for (int l = 0; l < C; l++) sum += red[l][tid];
    p.partials[tile * NQ + tid] = sum;
  }
}

template <int LOGN, bool CONTIG>
__device__ __forceinline__ void load(const cx<double>* in, int log_inner, int64_t tile, cx<double> (&v)[8]) {
  int64_t step;
  const cx<double>* q = in + Tile<LOGN, CONTIG>(nullptr).base(log_inner, tile, step);
#pragma unroll
  for (int k = 0; k < 8; k++) v[k] = q[k * step];
}

// Three blocks per SM (80 registers); with four (64, and x spilled) the step at 256^3 takes
// 994 us against 960, at 1024 x 1024 80 against 74.
template <int LOGN, bool CONTIG>
__global__ void __launch_bounds__(256, 3) k_pass_fx(const PassParams<double> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  cx<double> v[8];
  load<LOGN, CONTIG>(p.in, p.log_inner, blockIdx.x, v);
  pass<LOGN, CONTIG, false>(p, smem_raw, blockIdx.x, v);
}

// With the observable sums of the tile. A record of the 256^3 barrier (its three or four
// passes, with the FP64 butterflies before) cost 1.5 + 1.1 ms for the two passes that form
// sums; the run of 20 steps and 2 records takes 20.6 ms with these, about 23 before.
template <int LOGN, bool CONTIG>
__global__ void __launch_bounds__(256, 3) k_pass_fx_obs(const PassParams<double> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  cx<double> v[8];
  load<LOGN, CONTIG>(p.in, p.log_inner, blockIdx.x, v);
  if ((p.flags & (F_IFFT | F_PHASE | F_FFT | F_KIN)) || !(p.flags & F_NO_STORE))
    if (!pass<LOGN, CONTIG, true>(p, smem_raw, blockIdx.x, v)) return;
  obs_sums<LOGN, CONTIG>(p, smem_raw, blockIdx.x, v);
}

}  // namespace fxp
}  // namespace wp
