// Passes of the complex128 form in 64-bit fixed point (wp_fx.h): each line of a tile is held as
// integers with one exponent through the transforms and factors of the pass. Tiles and stage plan are
// those of the fixed-shape kernels of wp_kernels.cuh (2048 points, 256
// threads, n = 32..2048, the lengths whose stages unroll); those that form observable sums
// add them up in FP64 from the results; passes that apply a grid potential stay in FP64.
//
// Bound by the integer pipe (64 lanes per clock; ncu on 256^3: 66-72 % busy, FP64 before
// 92 %) and by instruction issue (65-68 %). Measured on the 256^3 barrier, CUDA events in the
// step, FP64 before, fixed point with the whole tile in shared memory, in registers with one
// exponent per tile, and these: FFT-only pass 617, 162, 159, 162 us; kinetic pass 1411, 333, 322,
// 330; potential pass 1118, 352, 290, 265 (its lines lie within a warp: no block barrier). The FP64 pipe bounds the
// sums of a record (86 % busy in the position sums, 488 us).
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

struct Max {
  static __device__ __forceinline__ uint32_t two(uint32_t a, uint32_t b) { return max(a, b); }
  static __device__ __forceinline__ uint32_t warp(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
};
struct Or {
  static __device__ __forceinline__ uint32_t two(uint32_t a, uint32_t b) { return a | b; }
  static __device__ __forceinline__ uint32_t warp(uint32_t v) { return __reduce_or_sync(0xffffffffu, v); }
};
struct Add {
  static __device__ __forceinline__ uint32_t two(uint32_t a, uint32_t b) { return a + b; }
  static __device__ __forceinline__ uint32_t warp(uint32_t v) { return __reduce_add_sync(0xffffffffu, v); }
};

// The shifts of a schedule's stages, two bits each.
__device__ __forceinline__ uint32_t packed(const FxSchedule& sc) {
  return sc.at[0] | (sc.at[1] << 2) | (sc.at[2] << 4) | (sc.at[3] << 6);
}

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

  // Reductions over the threads of a line. Where they are lanes of one warp (contiguous axes
  // up to 256 points) it is done in it; else the warps' parts cross shared memory (red: 256
  // words, not used by anything else between the barriers before and after the call).
  static constexpr bool IN_WARP = CONTIG && TL <= 32;
  template <class Op>
  static __device__ __forceinline__ uint32_t warp_part(uint32_t v) {
    if constexpr (CONTIG && TL >= 32) {
      v = Op::warp(v);
    } else {
#pragma unroll
      for (int o = CONTIG ? 1 : C; o < (CONTIG ? TL : 32); o <<= 1) v = Op::two(v, __shfl_xor_sync(0xffffffffu, v, o));
    }
    return v;
  }
  static __device__ __forceinline__ void put(uint32_t v, uint32_t* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if constexpr (CONTIG) {
      if (lane == 0) red[warp] = v;
    } else {
      if (lane < C) red[warp * 32 + lane] = v;
    }
  }
  template <class Op>
  static __device__ __forceinline__ uint32_t get(const uint32_t* red) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t v = 0;
    if constexpr (CONTIG) {
      constexpr int WL = TL < 32 ? 1 : TL / 32;  // warps of a line
#pragma unroll
      for (int k = 0; k < WL; k++) v = Op::two(v, red[(warp & ~(WL - 1)) + k]);
    } else {
      // every warp meets every column; of 64 columns odd and even warps one half each
#pragma unroll
      for (int k = 0; k < 8; k += C > 32 ? 2 : 1)
        v = Op::two(v, red[(k + (C > 32 ? warp & 1 : 0)) * 32 + (lane & (C - 1))]);
    }
    return v;
  }
  static __device__ __forceinline__ void line_max(uint32_t& m, uint32_t* red) {
    m = warp_part<Max>(m);
    if constexpr (!IN_WARP) {
      put(m, red);
      __syncthreads();
      m = get<Max>(red);
    }
  }
  static __device__ __forceinline__ void line_sum(uint32_t& L, uint32_t* red) {
    L = warp_part<Add>(L);
    if constexpr (!IN_WARP) {
      put(L, red);
      __syncthreads();
      L = get<Add>(red);
    }
  }
  // (union, sum) of the line's (any, L)
  static __device__ __forceinline__ void line_bounds(uint32_t& any, uint32_t& L, uint32_t* ra, uint32_t* rl) {
    any = warp_part<Or>(any);
    L = warp_part<Add>(L);
    if constexpr (!IN_WARP) {
      put(any, ra);
      put(L, rl);
      __syncthreads();
      any = get<Or>(ra);
      L = get<Add>(rl);
    }
  }

  // The forward transform of the line, with the shifts of its schedule (packed). The inverse one is the
  // same on points with real and imaginary parts exchanged, before and after.
  template <int LOGNS = 0, int S = 0>
  __device__ __forceinline__ void fft(cx<int64_t> (&x)[8], const FxRec* __restrict__ tw, uint32_t shifts) const {
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
        const uint32_t sh = (shifts >> (2 * S)) & 3u;
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
      fft<LOGNS + LR, S + 1>(x, tw, shifts);
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

// v: the thread's points, loaded by the caller. OBS: v returns the pass's results as doubles,
// for the sums.
template <int LOGN, bool CONTIG, bool OBS>
__device__ __forceinline__ void pass(const PassParams<double>& p, void* smem, int64_t tile, cx<double> (&v)[8]) {
  using TI = Tile<LOGN, CONTIG>;
  constexpr int TL = TI::TL;
  __shared__ uint32_t red[TI::IN_WARP ? 1 : 4][TI::IN_WARP ? 1 : 256];
  constexpr int R1 = TI::IN_WARP ? 0 : 1, R2 = 2 * R1, R3 = 3 * R1;
  const TI ti(smem);
  const uint32_t f = p.flags;
  const FxRec* tw = reinterpret_cast<const FxRec*>(p.Wln);
  const bool in_fx = (f & F_IN_FX) && p.fx_state, out_fx = (f & F_OUT_FX) && p.fx_state;

  // Load: the line's exponent (the largest leading bit), its bounds M and S, the integers.
  // An integer x of the line stands for x 2^(ex - 1085). A line that is all zero stays so; a
  // value that is not finite spoils its line.
  int32_t ex;
  uint32_t shifts, L = 0, any = 0, m = 0;
  enum { FINITE, ZERO, SPOIL } kind = FINITE;
  const bool ph = CONTIG && (f & F_PHASE), kin = !CONTIG && (f & F_KIN);
  bool swap = (f & F_IFFT) != 0;  // whether the points have their parts exchanged
  cx<int64_t> x[8];
  if (in_fx) {
#pragma unroll
    for (int k = 0; k < 8; k++) m = max(m, fx_code(wlo(v[k].re), wlo(v[k].im)));
    ti.line_max(m, red[0]);
    kind = m == 0u ? ZERO : m == (uint32_t)kFxNan ? SPOIL : FINITE;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t d = m - fx_code(wlo(v[k].re), wlo(v[k].im));
      L += fx_mag_int<kFxPassSum>(fx_shr64(absh(whi(v[k].re)), 0u, d)) +
           fx_mag_int<kFxPassSum>(fx_shr64(absh(whi(v[k].im)), 0u, d));
    }
    ti.line_sum(L, red[R1]);
    // the largest points have their leading bit at 62
    const FxSchedule sc = fx_schedule<LOGN>(64, fx_sum_bits<kFxPassSum>(L));
    ex = (int32_t)m - kFxBias + sc.total;  // that of the transform's results
    shifts = packed(sc);
    const uint32_t right = sc.first > 0 ? (uint32_t)sc.first : 0u, left = sc.first < 0 ? (uint32_t)-sc.first : 0u;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rl = wlo(v[k].re), il = wlo(v[k].im), c = fx_code(rl, il), d = m - c + right, jam = min(c, 1u);
      x[k] = mk((int64_t)((uint64_t)fx_align(rl, (int32_t)whi(v[k].re), d, jam) << left),
                (int64_t)((uint64_t)fx_align(il, (int32_t)whi(v[k].im), d, jam) << left));
    }
  } else {
#pragma unroll
    for (int k = 0; k < 8; k++) m = max(m, max(whi(v[k].re) & 0x7fffffffu, whi(v[k].im) & 0x7fffffffu));
    ti.line_max(m, red[0]);
    // all below 2^-953: lifted off the denormals, whose exponent field stands for 1
    const bool low = m < (70u << 20);
    uint32_t E = m >> 20;
    if (low) {
      E = max(E, 1u) + 900u;
#pragma unroll
      for (int k = 0; k < 8; k++) {
        any |= wlo(v[k].re) | wlo(v[k].im);
        v[k] = mk(v[k].re * 0x1p900, v[k].im * 0x1p900);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) {
      L += fx_mag<kFxPassSum>(whi(v[k].re), E - ((whi(v[k].re) >> 20) & 0x7ffu));
      L += fx_mag<kFxPassSum>(whi(v[k].im), E - ((whi(v[k].im) >> 20) & 0x7ffu));
    }
    ti.line_bounds(any, L, red[R1], red[R2]);
    kind = (m | any) == 0u ? ZERO : m >= 0x7ff00000u ? SPOIL : FINITE;
    const FxSchedule sc = fx_schedule<LOGN>(64, fx_sum_bits<kFxPassSum>(L));
    const uint32_t E2 = E + (uint32_t)sc.first;
    ex = (int32_t)E + sc.total - (low ? 900 : 0);
    shifts = packed(sc);
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
  const bool t0 = kin || (f & F_IFFT), t1 = kin || (f & F_FFT), mid = ph || kin || (t0 && t1);
#pragma unroll 1
  for (int it = 0; it < 2; it++) {
    if (it == 0 ? t0 : t1) ti.fft(x, tw, shifts);
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
    any = bad ? 0x80000000u : 0u;  // a factor that is not finite spoils its line
    L = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t ar = absh(x[k].re), ai = absh(x[k].im);
      any |= ar | ai;
      L += fx_mag_int<kFxPassSum>(ar) + fx_mag_int<kFxPassSum>(ai);
    }
    ti.line_bounds(any, L, red[R3], red[0]);
    if (any >> 31) kind = SPOIL;
    if (t0 && t1) {
      // the transform before has changed the bounds: a new scale
      const FxSchedule sc = fx_schedule<LOGN>(65 - __clz((int)(any & 0x7fffffffu)), fx_sum_bits<kFxPassSum>(L));
      ex += sc.total;
      shifts = packed(sc);
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = mk(shift_jam(x[k].re, sc.first), shift_jam(x[k].im, sc.first));
    }
    swap = kin;
    if (swap) exchange(x);
  }
  if (swap) exchange(x);
  if (kin) ex -= p.g.ln[0] + p.g.ln[1] + p.g.ln[2];  // 1/N
  // what a line that is all zero, or not finite, is stored with
  if (kind == ZERO) {
    ex = -2 * kFxNan;
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = mk((int64_t)0, (int64_t)0);
  }
  if (kind == SPOIL) ex = 2 * kFxNan;
  int64_t step;
  cx<double>* dst = p.out + ti.base(p.log_inner, tile, step);
  if (!OBS && out_fx) {
    // each point shifted up as far as it goes, so that the code bits cost nothing of it
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t up = (uint32_t)__clz((int)(absh(x[k].re) | absh(x[k].im))) - 1u;  // |x| < 2^63
      const int32_t code = min(max(ex + kFxBias - (int32_t)up, 0), kFxNan);
      const uint64_t re = (uint64_t)x[k].re << up, im = (uint64_t)x[k].im << up;
      const uint32_t rl = ((uint32_t)re & ~63u) | ((uint32_t)code >> 6), il = ((uint32_t)im & ~63u) | ((uint32_t)code & 63u);
      dst[k * step] = mk(__hiloint2double((int)(re >> 32), (int)rl), __hiloint2double((int)(im >> 32), (int)il));
    }
    return;
  }
  const bool chk = ex < 200 || ex > 1900;  // the range of a double may be left
#pragma unroll
  for (int k = 0; k < 8; k++) {
    uint32_t rh, rl, ih, il;
    fx_to_double(x[k].re, ex, rh, rl);
    fx_to_double(x[k].im, ex, ih, il);
    cx<double> y = mk(__hiloint2double((int)rh, (int)rl), __hiloint2double((int)ih, (int)il));
    if (chk) y = scaled(x[k], ex - 1085);
    if (kind == SPOIL) y = mk(__longlong_as_double(0x7ff8000000000000ll), __longlong_as_double(0x7ff8000000000000ll));
    if (!OBS || !(f & F_NO_STORE)) dst[k * step] = y;
    if (OBS) v[k] = y;
  }
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

// Three blocks per SM (80 registers); with four (64, and x spilled) the step at 256^3 took
// 994 us against 960, at 1024 x 1024 80 against 74 (with one exponent per tile).
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
    pass<LOGN, CONTIG, true>(p, smem_raw, blockIdx.x, v);
  obs_sums<LOGN, CONTIG>(p, smem_raw, blockIdx.x, v);
}

}  // namespace fxp
}  // namespace wp
