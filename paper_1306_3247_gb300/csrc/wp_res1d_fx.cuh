// Resident 1-D lines of the complex128 form in 64-bit fixed point (wp_fx.h): one block holds
// a line of n = 2^LOGN points (2^8 .. 2^13) for a chunk of steps, as k_res1d_fixed does for
// the other forms.
//
// The FP64 kernel was bound by the one FP64 pipe of its SM (one warp instruction every 19
// clocks): 33 us per step at 1024 points, 116 us at 4096. Here the transforms and factors
// are integer work, and the little FP64 work that is left per step (the coefficients f(t)
// and the cosines and sines of the plane-wave tables, a chain of about 5000 clocks) belongs
// to four warps of its own, which form the tables of the next potential phase while the
// others transform.
//
// Thread t holds the points t + k n/8, k = 0..7, in registers. These are the points of
// its butterfly in the first stage and of its outputs in the last one, so a transform goes
// through shared memory only between stages, and the factors between two transforms not at
// all. Shared memory is padded by one point in eight (the first stage writes eight
// consecutive points per thread).
#pragma once

#include "wp_fx_pass.cuh"

namespace wp {
namespace r1fx {

template <int LOGN>
struct Shape {
  static constexpr int N = 1 << LOGN, NT = N / 8, NW = NT / 32;
  // table warps, where the block has room for them
  static constexpr int TW = LOGN <= 12 ? 128 : 0;
  static constexpr int NHI = N > 64 ? N / 64 : 1;
  static constexpr size_t SMEM = (size_t)(N + N / 8) * sizeof(cx<int64_t>) + 2 * (size_t)(NHI + 64) * sizeof(FxRec);
};

__device__ __forceinline__ int pad(int i) { return i + (i >> 3); }

// Barrier of the NT transforming threads.
template <int NT>
__device__ __forceinline__ void bar() {
  asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory");
}

// The block's line state that is the same in every thread.
template <int LOGN>
struct Line {
  using SH = Shape<LOGN>;
  cx<int64_t>* s;
  uint32_t (*red)[32];  // [3][32]
  int32_t ex;           // the integers stand for x 2^(ex - 1085)
  int t;

  __device__ __forceinline__ uint32_t all(uint32_t v, bool max_) const {
    v = max_ ? __reduce_max_sync(0xffffffffu, v) : __reduce_or_sync(0xffffffffu, v);
    if ((t & 31) == 0) red[0][t >> 5] = v;
    bar<SH::NT>();
    v = (t & 31) < SH::NW ? red[0][t & 31] : 0u;
    return max_ ? __reduce_max_sync(0xffffffffu, v) : __reduce_or_sync(0xffffffffu, v);
  }
  // The union of the threads' `any` and the sum of their L.
  __device__ __forceinline__ uint32_t sum(uint32_t L, uint32_t& any) const {
    any = __reduce_or_sync(0xffffffffu, any);
    L = __reduce_add_sync(0xffffffffu, L);
    if ((t & 31) == 0) {
      red[1][t >> 5] = L;
      red[2][t >> 5] = any;
    }
    bar<SH::NT>();
    const bool in = (t & 31) < SH::NW;
    any = __reduce_or_sync(0xffffffffu, in ? red[2][t & 31] : 0u);
    return __reduce_add_sync(0xffffffffu, in ? red[1][t & 31] : 0u);
  }

  __device__ __forceinline__ void shift(cx<int64_t> (&x)[8], int32_t k) const {
#pragma unroll
    for (int i = 0; i < 8; i++) x[i] = mk(fxp::shift_jam(x[i].re, k), fxp::shift_jam(x[i].im, k));
  }
  // Scale x for a transform (its bounds from the block), shifting it in place; bS: bits of
  // the line sum afterwards.
  __device__ __forceinline__ FxSchedule scale(cx<int64_t> (&x)[8], int32_t& bS) {
    uint32_t any = 0, L = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t ar = fxp::absh(x[k].re), ai = fxp::absh(x[k].im);
      any |= ar | ai;
      L += (ar >> 14) + (ai >> 14) + 2u;
    }
    L = sum(L, any);
    bS = 78 - __clz((int)L);  // units of 2^46
    constexpr int LS1 = fx_mid(LOGN) ? kFxMidLog : LOGN;
    const FxSchedule sc = fx_schedule<LOGN, 0, LS1>(65 - __clz((int)any), bS);
    ex += sc.first;
    shift(x, sc.first);
    bS -= sc.total;
    return sc;
  }
  // The same after the first stages, from the values they left and bS.
  __device__ __forceinline__ FxSchedule rescale(cx<int64_t> (&x)[8], int32_t bS) {
    uint32_t any = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) any |= fxp::absh(x[k].re) | fxp::absh(x[k].im);
    any = all(any, false);
    const FxSchedule sc = fx_schedule<LOGN, kFxMidLog, LOGN>(65 - __clz((int)any), bS);
    ex += sc.total;
    shift(x, sc.first);
    return sc;
  }

  template <int LOGNS>
  __device__ __forceinline__ void butterflies(cx<int64_t> (&x)[8], const FxRec* __restrict__ tw, uint32_t sh) const {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), R = 1 << LR, B = 8 / R, NS = 1 << LOGNS;
#pragma unroll
    for (int b = 0; b < B; b++) {
      cx<int64_t> v[R];
#pragma unroll
      for (int r = 0; r < R; r++) v[r] = x[b * R + r];
      if constexpr (LOGNS > 0) {
        const FxRec* e = tw + wp_stage_tw_offset(LOGN, LOGNS) + ((t + b * SH::NT) & (NS - 1)) * (R - 1);
        v[0] = mk(v[0].re >> (2u - sh), v[0].im >> (2u - sh));
#pragma unroll
        for (int r = 1; r < R; r++) v[r] = fx_cmul(v[r], e[r - 1], sh);
      }
      fx_dft<R>(v);
#pragma unroll
      for (int r = 0; r < R; r++) x[b * R + r] = v[r];
    }
  }
  // Stage LOGNS > 0, the T-th of its schedule: from shared memory to shared memory, or to the
  // registers (last).
  template <int LOGNS, int T>
  __device__ __forceinline__ void stages(cx<int64_t> (&x)[8], const FxRec* __restrict__ tw, FxSchedule sc, int32_t bS) {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), R = 1 << LR, B = 8 / R, NR = SH::N / R;
    constexpr bool last = LOGNS + LR == LOGN, mid = fx_mid(LOGN) && LOGNS + LR == kFxMidLog;
    bar<SH::NT>();
#pragma unroll
    for (int b = 0; b < B; b++)
#pragma unroll
      for (int r = 0; r < R; r++) x[b * R + r] = s[pad(t + b * SH::NT + r * NR)];
    butterflies<LOGNS>(x, tw, sc.at[T]);
    if constexpr (last) {
      // output r of butterfly b is point t + (b + B r) n/8
      cx<int64_t> y[8];
#pragma unroll
      for (int b = 0; b < B; b++)
#pragma unroll
        for (int r = 0; r < R; r++) y[b + B * r] = x[b * R + r];
#pragma unroll
      for (int k = 0; k < 8; k++) x[k] = y[k];
    } else {
      if constexpr (mid)
        sc = rescale(x, bS);  // its barrier: everyone has read
      else
        bar<SH::NT>();
#pragma unroll
      for (int b = 0; b < B; b++) {
        const int j = t + b * SH::NT;
        const int d0 = ((j >> LOGNS) << (LOGNS + LR)) + (j & ((1 << LOGNS) - 1));
#pragma unroll
        for (int r = 0; r < R; r++) s[pad(d0 + (r << LOGNS))] = x[b * R + r];
      }
      stages<LOGNS + LR, mid ? 0 : T + 1>(x, tw, sc, bS);
    }
  }
  // The forward transform, registers to registers. The inverse is the same with real and
  // imaginary parts exchanged before and after.
  __device__ __forceinline__ void fft(cx<int64_t> (&x)[8], const FxRec* __restrict__ tw) {
    int32_t bS;
    const FxSchedule sc = scale(x, bS);  // its barrier frees the shared memory
    ex += sc.total - sc.first;
    static_assert(wp_stage_radix_log(LOGN, 0) == 3, "the first stage is radix 8");
    butterflies<0>(x, tw, 2u);
#pragma unroll
    for (int r = 0; r < 8; r++) s[pad(8 * t + r)] = x[r];
    stages<3, 1>(x, tw, sc, bS);
  }
};

__device__ __forceinline__ cx<int64_t> swapped(cx<int64_t> v) { return mk(v.im, v.re); }

// The coefficients and the plane-wave tables of the potential phase at time t (tau: phase
// length), by threads q = 0 .. nq - 1; sync: their barrier.
template <int LOGN, class F>
__device__ __forceinline__ void tables(const Res1dParams<double>& p, double t, double tau, double* fco, FxRec* hiT,
                                       FxRec* loT, int q, int nq, F&& sync) {
  using SH = Shape<LOGN>;
  const DevPot& pot = *p.pot;
  if (q < pot.nterms) fco[q] = term_coef(pot.term[q], t);
  sync();
  if (p.plane_mask == 0) return;
  double beta = 0.0, gamma = 0.0;
  for (int k = 0; k < pot.nterms; k++) {
    if (!((p.plane_mask >> k) & 1u)) continue;
    const wp_pot_term& tm = pot.term[k];
    if (tm.shape == WP_SHAPE_LINEAR) {
      beta += fco[k] * tm.a[0];
      gamma += fco[k] * tm.a[0] * (tm.c0[0] + tm.v[0] * t);
    } else {
      gamma -= fco[k];
    }
  }
  const double th0 = tau * (beta * p.g.xmin[0] - gamma) / p.g.hbar;
  const double del = tau * beta * p.g.dx[0] / p.g.hbar;
  for (int k = q; k < SH::NHI + 64; k += nq) {
    const bool hi = k < SH::NHI;
    double sn, cs;
    sincos(hi ? -fma((double)(k << 6), del, th0) : -(double)(k - SH::NHI) * del, &sn, &cs);
    (hi ? hiT[k] : loT[k - SH::NHI]) = fx_rec_of(cs, sn);
  }
}

template <int LOGN>
__device__ __forceinline__ void body(const Res1dParams<double>& p, unsigned char* smem) {
  using SH = Shape<LOGN>;
  constexpr int N = SH::N, NT = SH::NT;
  __shared__ uint32_t red[3][32];
  __shared__ double redd[32][NQ];
  __shared__ double qp[NQ], qm[NQ];
  __shared__ double fco[2][WP_MAX_TERMS];
  __shared__ int spoil;
  cx<int64_t>* s = reinterpret_cast<cx<int64_t>*>(smem);
  FxRec* tab = reinterpret_cast<FxRec*>(smem + (size_t)(N + N / 8) * sizeof(cx<int64_t>));
  const int t = threadIdx.x;
  const int64_t s0 = p.ctrl->step, m = p.nsteps;
  const double dt = p.g.dt;
  const bool vkv = p.order == WP_ORDER_VKV;
  // Potential phases of the chunk, in order: VKV m + 1 of them (half, full, .., half), KVK m.
  const int64_t nphase = m > 0 ? (vkv ? m + 1 : m) : 0;
  auto phase_time = [&](int64_t k) { return p.g.t0 + (double)(s0 + k) * dt + (vkv ? 0.0 : 0.5 * dt); };
  auto phase_half = [&](int64_t k) { return vkv && (k == 0 || k == m); };
  auto hiT = [&](int64_t k) { return tab + (k & 1) * (SH::NHI + 64); };
  auto make = [&](int64_t k, int q, int nq, auto&& sync) {
    tables<LOGN>(p, phase_time(k), phase_half(k) ? 0.5 * dt : dt, fco[k & 1], hiT(k), hiT(k) + SH::NHI, q, nq, sync);
  };
  // one barrier of the whole block per phase: the tables of phase k are complete, and those
  // of phase k - 1 no longer read
  if (t == 0) spoil = 0;
  __syncthreads();
  if constexpr (SH::TW > 0) {
    if (t >= NT) {
      for (int64_t k = 0; k < nphase; k++) {
        make(k, t - NT, SH::TW, [] { asm volatile("bar.sync 2, %0;" ::"n"(SH::TW) : "memory"); });
        __syncthreads();
      }
      __syncthreads();
      return;
    }
  }
  // load
  Line<LOGN> ln{s, red, 0, t};
  cx<int64_t> x[8];
  bool zero;
  {
    cx<double> v[8];
    uint32_t mx = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) v[k] = p.psi[t + k * NT];
    auto top = [&] {
      uint32_t w = 0;
#pragma unroll
      for (int k = 0; k < 8; k++) w = max(w, max(fxp::whi(v[k].re) & 0x7fffffffu, fxp::whi(v[k].im) & 0x7fffffffu));
      return ln.all(w, true);
    };
    mx = top();
    int32_t off = 0;
    if (mx < (70u << 20)) {
      bar<NT>();
      off = -900;  // off the denormals
#pragma unroll
      for (int k = 0; k < 8; k++) v[k] = mk(v[k].re * 0x1p900, v[k].im * 0x1p900);
      mx = top();
    }
    zero = mx == 0u;
    if (mx >= 0x7ff00000u) spoil = 1;
    const uint32_t E = zero || mx >= 0x7ff00000u ? 1023u : mx >> 20;
    ln.ex = (int32_t)E + 1 + off;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const uint32_t rh = fxp::whi(v[k].re), ih = fxp::whi(v[k].im);
      x[k] = mk(fx_from_double(rh, fxp::wlo(v[k].re), E + 1u - ((rh >> 20) & 0x7ffu)),
                fx_from_double(ih, fxp::wlo(v[k].im), E + 1u - ((ih >> 20) & 0x7ffu)));
    }
  }
  int bad = 0;
  auto potential = [&](int64_t kph) {
    if constexpr (SH::TW == 0) {
      bar<NT>();
      make(kph, t, NT, [] { bar<NT>(); });
    }
    __syncthreads();
    const FxRec* hi = hiT(kph);
    const FxRec* lo = hi + SH::NHI;
    const double* fc = fco[kph & 1];
    const bool half = phase_half(kph);
    const double tau = half ? 0.5 * dt : dt, tm0 = phase_time(kph);
    const FxRec* S = p.Sfx[half ? 1 : 0];
    const DevPot& pot = *p.pot;
    const bool stat = p.static_mask != 0, plane = p.plane_mask != 0;
    int b = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const int i = t + k * NT;
      if (stat) {
        const FxRec w = S[i];
        b |= w.bad;
        x[k] = fx_cmul(x[k], w);
      }
      if (plane) {
        x[k] = fx_cmul(x[k], hi[i >> 6]);
        x[k] = fx_cmul(x[k], lo[i & 63]);
      }
    }
    if (plane) b |= hi[t % SH::NHI].bad | lo[t & 63].bad;
    if (p.gen_mask) {
      // not unrolled: the FP64 exponentials and sines are long code
#pragma unroll 1
      for (int k = 0; k < 8; k++) {
        const double xi = p.g.xmin[0] + (double)(t + k * NT) * p.g.dx[0];
        double V = 0.0;
        for (int e = 0; e < pot.nterms; e++) {
          if (!((p.gen_mask >> e) & 1u)) continue;
          const wp_pot_term& tm = pot.term[e];
          const double sh = (tm.shape == WP_SHAPE_GAUSS) ? gauss_axis_factor(tm, 0, xi, tm0) : term_axis_part(tm, 0, xi, tm0);
          V += fc[e] * sh;
        }
        double sn, cs;
        sincos(-V * tau / p.g.hbar, &sn, &cs);
        const FxRec w = fx_rec_of(cs, sn);
        b |= w.bad;
        // rotate through the registers, so that the loop indexes none of them
        const cx<int64_t> v = fx_cmul(x[0], w);
#pragma unroll
        for (int q = 0; q < 7; q++) x[q] = x[q + 1];
        x[7] = v;
      }
    }
    bad |= b;
  };
  auto kinetic = [&](int half) {
    const FxRec* K = p.Kfx[half];
    // forward, factor with the exchange for the inverse, inverse; one copy of the code
#pragma unroll 1
    for (int it = 0; it < 2; it++) {
      ln.fft(x, p.Wfx);
      if (it == 0) {
#pragma unroll
        for (int k = 0; k < 8; k++) {
          const FxRec w = K[t + k * NT];
          bad |= w.bad;
          x[k] = swapped(fx_cmul(x[k], w));
        }
      }
    }
#pragma unroll
    for (int k = 0; k < 8; k++) x[k] = swapped(x[k]);
    ln.ex -= LOGN;  // 1/N
  };
  // VKV: P K P .. K P; KVK: K P K .. P K. One call of each, so that their code is there once.
  if (m > 0) {
#pragma unroll 1
    for (int64_t k = 0; k <= m; k++) {
      if (vkv || k > 0) potential(vkv ? k : k - 1);
      if (!vkv || k < m) kinetic(!vkv && (k == 0 || k == m) ? 1 : 0);
    }
  }
  if (bad) spoil = 1;
  bar<NT>();
  const bool nan = spoil != 0;
  // store; position sums of the stored values
  const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  const bool chk = ln.ex < 200 || ln.ex > 1900;
  double acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) acc[q] = 0.0;
  auto value = [&](cx<int64_t> v) {
    uint32_t rh, rl, ih, il;
    fx_to_double(v.re, ln.ex, rh, rl);
    fx_to_double(v.im, ln.ex, ih, il);
    cx<double> y = mk(__hiloint2double((int)rh, (int)rl), __hiloint2double((int)ih, (int)il));
    if (chk) y = fxp::scaled(v, ln.ex - 1085);
    if (zero) y = mk(0.0, 0.0);
    if (nan) y = mk(qnan, qnan);
    return y;
  };
#pragma unroll
  for (int k = 0; k < 8; k++) {
    const int i = t + k * NT;
    const cx<double> v = value(x[k]);
    if (m > 0) p.psi[i] = v;
    if (p.obs) {
      // V = V_s + beta x - gamma + general terms: the plane part from the moments below
      const double rho = norm2(v), xi = p.g.xmin[0] + (double)i * p.g.dx[0];
      const double xr = xi * rho;
      acc[Q_RHO] += rho;
      acc[Q_X] += xr;
      acc[Q_XX] += xi * xr;
      acc[Q_V] += p.Vs[i] * rho;
      if (p.autocorr) {
        const cx<double> c = cmulc(v, p.psi0[i]);
        acc[Q_AC_RE] += c.re;
        acc[Q_AC_IM] += c.im;
      }
    }
  }
  if (p.obs) {
    const DevPot& pot = *p.pot;
    const double tm0 = p.g.t0 + (double)(s0 + m) * dt;
    if (t < pot.nterms) fco[0][t] = term_coef(pot.term[t], tm0);
    bar<NT>();
    if (p.gen_mask) {
      for (int k = 0; k < 8; k++) {
        const double xi = p.g.xmin[0] + (double)(t + k * NT) * p.g.dx[0];
        const cx<double> v = value(x[0]);
        double V = 0.0;
        for (int e = 0; e < pot.nterms; e++) {
          if (!((p.gen_mask >> e) & 1u)) continue;
          const wp_pot_term& tm = pot.term[e];
          V += fco[0][e] * ((tm.shape == WP_SHAPE_GAUSS) ? gauss_axis_factor(tm, 0, xi, tm0) : term_axis_part(tm, 0, xi, tm0));
        }
        acc[Q_V] += V * norm2(v);
        const cx<int64_t> first = x[0];
#pragma unroll
        for (int q = 0; q < 7; q++) x[q] = x[q + 1];
        x[7] = first;
      }
    }
    auto block_total = [&](double* out) {
#pragma unroll
      for (int q = 0; q < NQ; q++) {
        double v = acc[q];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        if ((t & 31) == 0) redd[t >> 5][q] = v;
      }
      bar<NT>();
      if (t < NQ) {
        double v = 0.0;
        for (int w = 0; w < SH::NW; w++) v += redd[w][t];
        out[t] = v;
      }
      bar<NT>();
    };
    block_total(qp);
    ln.fft(x, p.Wfx);
#pragma unroll
    for (int q = 0; q < NQ; q++) acc[q] = 0.0;
#pragma unroll
    for (int k = 0; k < 8; k++) {
      const double rho = norm2(value(x[k])), kk = wavenumber(p.g, 0, t + k * NT), kr = kk * rho;
      acc[Q_RHOK] += rho;
      acc[Q_K] += kr;
      acc[Q_K2] += kk * kr;
    }
    block_total(qm);
    if (t == 0) {
      for (int e = 0; e < pot.nterms; e++) {
        if (!((p.plane_mask >> e) & 1u)) continue;
        const wp_pot_term& tm = pot.term[e];
        if (tm.shape == WP_SHAPE_LINEAR)
          qp[Q_V] += fco[0][e] * tm.a[0] * (qp[Q_X] - (tm.c0[0] + tm.v[0] * tm0) * qp[Q_RHO]);
        else
          qp[Q_V] += fco[0][e] * qp[Q_RHO];
      }
      const int64_t slot = p.ctrl->nobs;
      if (slot < p.obs_cap) {
        finish_obs(qp, qm, p.g, N, p.autocorr, tm0, s0 + m, p.obs_out + slot * 16);
        if (!isfinite(p.obs_out[slot * 16 + 1])) p.ctrl->err = WP_ENONFINITE;
      }
      p.ctrl->nobs = slot + 1;
    }
  }
  if (t == 0) p.ctrl->step = s0 + m;
  if constexpr (SH::TW > 0) __syncthreads();
}

template <int LOGN>
__global__ void __launch_bounds__(Shape<LOGN>::NT + Shape<LOGN>::TW) k_res1d_fx(const Res1dParams<double> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  body<LOGN>(p, smem_raw);
}

// Block b runs instance b (all of one line length) for nsteps.
template <int LOGN>
__global__ void __launch_bounds__(Shape<LOGN>::NT + Shape<LOGN>::TW)
    k_res1d_fx_batch(const Res1dParams<double>* __restrict__ params, int64_t nsteps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) unsigned char raw[sizeof(Res1dParams<double>)];
  Res1dParams<double>& p = *reinterpret_cast<Res1dParams<double>*>(raw);
  const int* src = reinterpret_cast<const int*>(&params[blockIdx.x]);
  for (int k = threadIdx.x; k < (int)(sizeof(Res1dParams<double>) / sizeof(int)); k += blockDim.x)
    reinterpret_cast<int*>(raw)[k] = src[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    p.nsteps = nsteps;
    p.obs = 0;
  }
  __syncthreads();
  body<LOGN>(p, smem_raw);
}

}  // namespace r1fx
}  // namespace wp
