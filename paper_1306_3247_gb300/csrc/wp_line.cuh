// Resident 1-D lines of compile-time length n = 2^LOGN (2^8 .. 2^14): a line stays on chip for a
// chunk of steps, held by one block (batched instances, short lines) or by a cluster of R
// blocks (a long line on its own). One body serves both and the three arithmetic forms, so
// that an instance gives the same bits alone and in a batch.
//
// Points. Block c of the cluster holds the points i = c (mod R); its thread t those with
// i = c + R (t + k NT), k = 0 .. P - 1, in registers. These are the points of its butterflies in
// the first stage of a transform and the outputs of its butterflies in the last one, so the
// factors between two transforms never go through shared memory. Every stage but the first
// reads and writes points of one residue class mod R (R divides the spans 8, 64, ..): only the
// first stage's outputs cross the cluster, through distributed shared memory. They are
// announced on an mbarrier of the receiving block, one arrival per sending warp, which leaves
// the rest of the cluster alone. Two buffers, used in turn by successive transforms, let a
// block write to a neighbour that still reads the transform before: its next write to the
// same buffer follows a transform that needed every warp of that neighbour. Shared memory is
// padded by one point in eight (the first stage writes eight points per thread).
//
// complex128 lines are in 64-bit fixed point (wp_fx.h): in FP64 the one FP64 pipe of an SM
// bound them (one warp instruction every 19 clocks). The scale of a transform then takes the
// bounds of the whole line: one more exchange of a few words, or two from 2048 points on.
//
// Four warps of their own form the tables of the next potential phase (cosines and sines
// in FP64, a chain of about 5000 clocks) while the others transform; for the shortest lines
// that chain is the step.
//
// Measured, us per step of the driven trap alone (one block with its points in shared memory
// and FP64 arithmetic for complex128 before -> now): complex64 1024 points 7.2 -> 3.2, 4096
// 18.1 -> 4.2, 16384 54.1 -> 8.5; float-float 4096 33.4 -> 15.3, 8192 65.6 -> 21.6; complex128
// 1024 28.1 -> 6.8, 4096 111 -> 11.0, 8192 237 -> 12.7. The batch's 1-D launches (256 lines, 20
// steps, complex64) 1946 -> 1092 us. A cluster is bound by latency: shared memory, the
// exchange, barriers and integer or FP32 chains, with 2 to 8 warps per SM.
#pragma once

#include "wp_fx_pass.cuh"

namespace wp {
namespace line {

__device__ __forceinline__ int pad(int i) { return i + (i >> 3); }

// ------------------------------------------------------------------ cluster primitives
__device__ __forceinline__ uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address of p (this block's shared memory) in block `rank` of the cluster.
template <class V>
__device__ __forceinline__ uint32_t remote(const V* p, uint32_t rank) {
  uint32_t a = (uint32_t)__cvta_generic_to_shared(p), r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
__device__ __forceinline__ void remote_store(uint32_t a, cx<float> v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.re), "f"(v.im) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, cx<ff> v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.re.hi), "f"(v.re.lo), "f"(v.im.hi),
               "f"(v.im.lo)
               : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, cx<int64_t> v) {
  asm volatile("st.shared::cluster.v2.b64 [%0], {%1, %2};" ::"r"(a), "l"(v.re), "l"(v.im) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, uint32_t v) {
  asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void remote_store(uint32_t a, double v) {
  asm volatile("st.shared::cluster.f64 [%0], %1;" ::"r"(a), "d"(v) : "memory");
}
// Arrival on block `rank`'s mbarrier, after the calling thread's (and, past a __syncwarp, its
// warp's) stores to that block.
__device__ __forceinline__ void remote_arrive(uint64_t* bar, uint32_t rank) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(remote(bar, rank)) : "memory");
}
__device__ __forceinline__ bool try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}"
      : "=r"(done)
      : "r"((uint32_t)__cvta_generic_to_shared(bar)), "r"(parity)
      : "memory");
  return done != 0;
}

// ------------------------------------------------------------------ arithmetic of a form
// T: the handle's real type; V: a point in registers and shared memory; Rec: a factor.
template <class T>
struct Form {
  using V = cx<T>;
  using Rec = TwE<T>;
  static constexpr bool fixed_point = false;
  static __device__ __forceinline__ V mul(V v, const Rec& w) { return tw_apply<false>(v, w); }
  static __device__ __forceinline__ Rec rec(double c, double s) { return make_rec<T>(c, s); }
  static __device__ __forceinline__ const Rec* kinetic(const Res1dParams<T>& p, int half) { return p.Krec[half]; }
  static __device__ __forceinline__ const Rec* statics(const Res1dParams<T>& p, int half) { return p.S[half]; }
  static __device__ __forceinline__ int bad(const Rec&) { return 0; }
};
template <>
struct Form<double> {
  using V = cx<int64_t>;
  using Rec = FxRec;
  static constexpr bool fixed_point = true;
  static __device__ __forceinline__ V mul(V v, const Rec& w) { return fx_cmul(v, w); }
  static __device__ __forceinline__ Rec rec(double c, double s) { return fx_rec_of(c, s); }
  static __device__ __forceinline__ const Rec* kinetic(const Res1dParams<double>& p, int half) { return p.Kfx[half]; }
  static __device__ __forceinline__ const Rec* statics(const Res1dParams<double>& p, int half) { return p.Sfx[half]; }
  static __device__ __forceinline__ int bad(const Rec& w) { return w.bad; }
};

// Shape of the kernel of a length and cluster size R = 2^LOGR; BATCH: one of many lines.
template <class T, int LOGN, int LOGR, bool BATCH = false>
struct Shape {
  using F = Form<T>;
  static constexpr int N = 1 << LOGN, R = 1 << LOGR;
  static constexpr int P = 8;  // points per thread
  static constexpr int NT = N / (P * R), NW = NT / 32;
  // Threads of their own for the tables, except in blocks of a batch that fill the SM in pairs:
  // there the other block's work hides the tables, and the registers are worth more.
  static constexpr int TW = BATCH && NT >= 256 ? 0 : 128;
  static constexpr int MIN_BLOCKS = BATCH && NT == 512 ? 2 : 1;
  // plane-wave phase of point i: coarse entry i >> LOGLO times fine entry i mod 2^LOGLO
  static constexpr int LOGLO = LOGN >= 13 ? 7 : 6, NLO = 1 << LOGLO, NHI = N >> LOGLO;
  static constexpr int NBUF = R > 1 ? 2 : 1;
  static constexpr int LINE = N / R + N / R / 8;  // points of a padded buffer
  static constexpr size_t TAB = 2 * (size_t)(NHI + NLO) * sizeof(typename F::Rec);
  // a cluster's block copies its residue class of the twiddles (N / R records at most): in the
  // common table they lie R records apart
  static constexpr bool OWN = R > 1 && !BATCH;
  static constexpr size_t TWID = OWN ? (size_t)N / R * sizeof(typename F::Rec) : 0;
  static constexpr size_t SMEM = NBUF * (size_t)LINE * sizeof(typename F::V) + TAB + TWID;
  // the factors of the full steps stay in registers for the chunk, where there are enough
  static constexpr bool KEEP = R > 1 && !BATCH;
};

// The line as a thread sees it.
template <class T, int LOGN, int LOGR, bool BATCH>
struct Line {
  using SH = Shape<T, LOGN, LOGR, BATCH>;
  using F = Form<T>;
  using V = typename F::V;
  using Rec = typename F::Rec;
  static constexpr int R = SH::R, P = SH::P, NT = SH::NT;
  V* s;                  // buffers
  uint32_t (*red)[32];   // [2][32]: block reductions
  uint32_t (*cred)[2][8];  // [2]: the cluster's
  uint64_t* mb;          // mbarriers: [0..1] buffers, [2..3] cluster reductions, [4..5] records
  Ctrl* ctrl;
  int32_t ex;            // fixed point: an integer x stands for x 2^(ex - 1085)
  int t;
  uint32_t c;            // rank in the cluster
  uint32_t nfft, nred;   // exchanges so far: buffer n & 1, phase parity (n >> 1) & 1
  bool lost;             // a wait has run out: the rest of the chunk no longer waits, and the thread's points are lost

  __device__ __forceinline__ int point(int k) const { return (int)c + R * (t + k * NT); }
  // Barrier of the block's transforming threads.
  static __device__ __forceinline__ void bar() { asm volatile("bar.sync 1, %0;" ::"n"(NT) : "memory"); }

  // Waits for the n-th use of a pair of mbarriers, a second or so at most.
  __device__ __forceinline__ void wait(uint64_t* pair, uint32_t n) {
    if (lost) return;
    for (int k = 0; k < (1 << 20); k++)
      if (try_wait(pair + (n & 1u), (n >> 1) & 1u)) return;
    lost = true;
    ctrl->lost = 1;
  }

  // (union, sum) of the line's (any, L), in every thread.
  __device__ __forceinline__ void reduce(uint32_t& any, uint32_t& L, bool max_ = false) {
    auto comb = [&](uint32_t v) {
      return max_ ? __reduce_max_sync(0xffffffffu, v) : __reduce_or_sync(0xffffffffu, v);
    };
    any = comb(any);
    L = __reduce_add_sync(0xffffffffu, L);
    if ((t & 31) == 0) {
      red[0][t >> 5] = any;
      red[1][t >> 5] = L;
    }
    bar();
    const bool in = (t & 31) < SH::NW;
    any = comb(in ? red[0][t & 31] : 0u);
    L = __reduce_add_sync(0xffffffffu, in ? red[1][t & 31] : 0u);
    if constexpr (R > 1) {
      if (t < R) {
        remote_store(remote(&cred[nred & 1u][0][c], (uint32_t)t), any);
        remote_store(remote(&cred[nred & 1u][1][c], (uint32_t)t), L);
        remote_arrive(mb + 2 + (nred & 1u), (uint32_t)t);
      }
      __syncwarp();
      wait(mb + 2, nred);
      __syncwarp();
      any = comb((t & 31) < R ? cred[nred & 1u][0][t & 31] : 0u);
      L = __reduce_add_sync(0xffffffffu, (t & 31) < R ? cred[nred & 1u][1][t & 31] : 0u);
      nred++;
    }
  }

  // ---- fixed point: scaling
  __device__ __forceinline__ void shift(V (&x)[P], int32_t k) const {
    if constexpr (F::fixed_point)
#pragma unroll
      for (int i = 0; i < P; i++) x[i] = mk(fxp::shift_jam(x[i].re, k), fxp::shift_jam(x[i].im, k));
  }
  // x scaled for a transform by the line's bounds; bS: bits of the line sum afterwards.
  __device__ __forceinline__ FxSchedule scale(V (&x)[P], int32_t& bS) {
    uint32_t any = 0, L = 0;
#pragma unroll
    for (int k = 0; k < P; k++) {
      const uint32_t ar = fxp::absh(x[k].re), ai = fxp::absh(x[k].im);
      any |= ar | ai;
      L += fx_mag_int<kFxLineSum>(ar) + fx_mag_int<kFxLineSum>(ai);
    }
    reduce(any, L);
    bS = fx_sum_bits<kFxLineSum>(L);
    constexpr int LS1 = fx_mid(LOGN) ? kFxMidLog : LOGN;
    const FxSchedule sc = fx_schedule<LOGN, 0, LS1>(65 - __clz((int)any), bS);
    ex += sc.total;
    shift(x, sc.first);
    bS -= sc.total;
    return sc;
  }
  // The same after the first stages, from the values they left and bS.
  __device__ __forceinline__ FxSchedule rescale(V (&x)[P], int32_t bS) {
    uint32_t any = 0, L = 0;
#pragma unroll
    for (int k = 0; k < P; k++) any |= fxp::absh(x[k].re) | fxp::absh(x[k].im);
    reduce(any, L);
    const FxSchedule sc = fx_schedule<LOGN, kFxMidLog, LOGN>(65 - __clz((int)any), bS);
    ex += sc.total;
    shift(x, sc.first);
    return sc;
  }

  // ---- transform
  template <int LOGNS, bool INV>
  __device__ __forceinline__ void butterflies(V (&x)[P], const Rec* __restrict__ tw, uint32_t sh) const {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), RX = 1 << LR, B = P / RX, NS = 1 << LOGNS;
#pragma unroll
    for (int b = 0; b < B; b++) {
      V v[RX];
#pragma unroll
      for (int r = 0; r < RX; r++) v[r] = x[b + B * r];
      if constexpr (LOGNS > 0) {
        // twiddle r of the stage at (r - 1) NS + jm, or that divided by R (jm = c mod R)
        constexpr int LT = SH::OWN ? LOGR : 0;
        const Rec* e = tw + (wp_stage_tw_offset(LOGN, LOGNS) >> LT) + ((point(b) & (NS - 1)) >> LT);
        if constexpr (F::fixed_point) {
          v[0] = mk(v[0].re >> (2u - sh), v[0].im >> (2u - sh));
#pragma unroll
          for (int r = 1; r < RX; r++) v[r] = fx_cmul(v[r], e[(r - 1) * (NS >> LT)], sh);
        } else {
#pragma unroll
          for (int r = 1; r < RX; r++) v[r] = tw_apply<INV>(v[r], e[(r - 1) * (NS >> LT)]);
        }
      }
      if constexpr (F::fixed_point)
        fx_dft<RX>(v);
      else
        Dft<T, RX, INV>::run(v);
#pragma unroll
      for (int r = 0; r < RX; r++) x[b + B * r] = v[r];
    }
  }
  // Stage LOGNS > 0, the TI-th of its schedule: butterfly b of the thread reads the points
  // point(b) + r n/RX, and leaves its outputs in shared memory, or (last stage) in x.
  template <int LOGNS, int TI, bool INV>
  __device__ __forceinline__ void stages(V (&x)[P], V* s, const Rec* __restrict__ tw, FxSchedule sc, int32_t bS) {
    constexpr int LR = wp_stage_radix_log(LOGN, LOGNS), RX = 1 << LR, B = P / RX;
    constexpr bool last = LOGNS + LR == LOGN;
    constexpr bool mid = F::fixed_point && fx_mid(LOGN) && LOGNS + LR == kFxMidLog;
#pragma unroll
    for (int b = 0; b < B; b++)
#pragma unroll
      for (int r = 0; r < RX; r++) x[b + B * r] = s[pad(t + b * NT + r * (SH::N / RX / R))];
    butterflies<LOGNS, INV>(x, tw, F::fixed_point ? sc.at[TI] : 0u);
    if constexpr (!last) {
      if constexpr (mid)
        sc = rescale(x, bS);  // its barrier: everyone has read
      else
        bar();
#pragma unroll
      for (int b = 0; b < B; b++) {
        const int j = point(b);
        const int d0 = (((j >> LOGNS) << (LOGNS + LR)) + (j & ((1 << LOGNS) - 1))) >> LOGR;
#pragma unroll
        for (int r = 0; r < RX; r++) s[pad(d0 + (r << (LOGNS - LOGR)))] = x[b + B * r];
      }
      bar();
      stages<LOGNS + LR, mid ? 0 : TI + 1, INV>(x, s, tw, sc, bS);
    }
  }
  // The transform, registers to registers. Fixed point: forward only (the inverse is the same
  // with real and imaginary parts exchanged before and after).
  template <bool INV>
  __device__ __forceinline__ void fft(V (&x)[P], const Rec* __restrict__ tw) {
    static_assert(wp_stage_radix_log(LOGN, 0) == 3, "the first stage is radix 8");
    int32_t bS = 0;
    FxSchedule sc = {};
    if constexpr (F::fixed_point) sc = scale(x, bS);
    butterflies<0, INV>(x, tw, 2u);
    constexpr int B = P / 8;
    if constexpr (R == 1) {
      if constexpr (!F::fixed_point) bar();  // the reads of the transform before are done
#pragma unroll
      for (int b = 0; b < B; b++)
#pragma unroll
        for (int r = 0; r < 8; r++) s[pad(8 * point(b) + r)] = x[b + B * r];
      bar();
      stages<3, 1, INV>(x, s, tw, sc, bS);
    } else {
      V* buf = s + (nfft & 1u) * SH::LINE;
#pragma unroll
      for (int b = 0; b < B; b++)
#pragma unroll
        for (int r = 0; r < 8; r++)
          remote_store(remote(&buf[pad((8 * point(b) + r) >> LOGR)], (uint32_t)(r & (R - 1))), x[b + B * r]);
      __syncwarp();
      if ((t & 31) < R) remote_arrive(mb + (nfft & 1u), (uint32_t)(t & 31));
      __syncwarp();
      wait(mb, nfft);
      __syncwarp();
      nfft++;
      stages<3, 1, INV>(x, buf, tw, sc, bS);
    }
  }
};

__device__ __forceinline__ cx<int64_t> swapped(cx<int64_t> v) { return mk(v.im, v.re); }

// The coefficients and the plane-wave tables of the potential phase at time t (tau_hbar: phase
// length / hbar), by threads q = 0 .. nq - 1; sync: their barrier. A block of a cluster needs the fine
// entries k = c (mod R) only.
template <class T, class SH, class S>
__device__ __forceinline__ void tables(const Res1dParams<T>& p, double t, double tau_hbar, double* fco,
                                       typename Form<T>::Rec* hiT, uint32_t c, int q, int nq, S&& sync) {
  using F = Form<T>;
  constexpr int R = SH::R, NL = SH::NLO / R;
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
  const double th0 = tau_hbar * (beta * p.g.xmin[0] - gamma);
  const double del = tau_hbar * (beta * p.g.dx[0]);
  for (int e = q; e < SH::NHI + NL; e += nq) {
    const bool hi = e < SH::NHI;
    const int k = hi ? e : (e - SH::NHI) * R + (int)c;
    double sn, cs;
    sincos(hi ? -fma((double)(k << SH::LOGLO), del, th0) : -(double)k * del, &sn, &cs);
    hiT[hi ? k : SH::NHI + k] = F::rec(cs, sn);
  }
}

// Thread q's part of the coefficients at time t (one copy of the sine's code beside the tables').
static __device__ __noinline__ void record_coefs(const DevPot& pot, double t, double* fco, int q) {
  if (q < pot.nterms) fco[q] = term_coef(pot.term[q], t);
}

// FP64 sums of the line in a fixed order into `out` (shared memory of block 0): the block's
// warps in order, then (part: [R][NQ] in block 0, n: which of its two record mbarriers) the
// blocks. used: the quantities to sum (a shuffle tree is five dependent FP64 adds, 320 clocks,
// for each).
template <class LN>
__device__ __forceinline__ void total(LN& ln, double (&acc)[NQ], uint32_t used, double (*redd)[NQ], double (*part)[NQ],
                                      int n, double* out) {
  const int t = ln.t;
#pragma unroll
  for (int q = 0; q < NQ; q++) {
    double v = 0.0;
    if ((used >> q) & 1u) {
      v = acc[q];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    }
    if ((t & 31) == 0) redd[t >> 5][q] = v;
  }
  ln.bar();
  if (t < NQ) {
    double v = redd[0][t];
    for (int w = 1; w < LN::SH::NW; w++) v += redd[w][t];
    if constexpr (LN::R == 1)
      out[t] = v;
    else
      remote_store(remote(&part[ln.c][t], 0u), v);
  }
  if constexpr (LN::R > 1) {
    __syncwarp();
    if (t == 0) remote_arrive(ln.mb + 4 + n, 0u);
    __syncwarp();
    if (ln.c == 0u) {
      ln.wait(ln.mb + 4 + n, 0u);
      __syncwarp();
      if (t < NQ) {
        double v = part[0][t];
        for (int b = 1; b < LN::R; b++) v += part[b][t];
        out[t] = v;
      }
    }
  }
  ln.bar();
}

template <class T, int LOGN, int LOGR, bool BATCH>
__device__ __forceinline__ void body(const Res1dParams<T>& p, unsigned char* smem) {
  using SH = Shape<T, LOGN, LOGR, BATCH>;
  using F = Form<T>;
  using LN = Line<T, LOGN, LOGR, BATCH>;
  using V = typename F::V;
  using Rec = typename F::Rec;
  constexpr int N = SH::N, R = SH::R, P = SH::P, NT = SH::NT;
  __shared__ uint32_t red[2][32];
  __shared__ uint32_t cred[2][2][8];
  __shared__ double redd[32][NQ], part[2][R > 1 ? R : 1][NQ];
  __shared__ double qp[NQ], qm[NQ];
  __shared__ double fco[2][WP_MAX_TERMS];
  __shared__ __align__(8) uint64_t mb[6];
  V* s = reinterpret_cast<V*>(smem);
  Rec* tab = reinterpret_cast<Rec*>(smem + SH::NBUF * (size_t)SH::LINE * sizeof(V));
  const int t = threadIdx.x;
  const uint32_t c = R > 1 ? cluster_rank() : 0u;
  const int64_t s0 = p.ctrl->step, m = p.nsteps;
  const double dt = p.g.dt;
  const bool vkv = p.order == WP_ORDER_VKV;
  // Potential phases of the chunk, in order: VKV m + 1 of them (half, full, .., half), KVK m.
  const int64_t nphase = m > 0 ? (vkv ? m + 1 : m) : 0;
  auto phase_time = [&](int64_t k) { return p.g.t0 + (double)(s0 + k) * dt + (vkv ? 0.0 : 0.5 * dt); };
  auto phase_half = [&](int64_t k) { return vkv && (k == 0 || k == m); };
  auto hiT = [&](int64_t k) { return tab + (k & 1) * (SH::NHI + SH::NLO); };
  const double tau_hbar = dt / p.g.hbar;
  auto make = [&](int64_t k, int q, int nq, auto&& sync) {
    tables<T, SH>(p, phase_time(k), phase_half(k) ? 0.5 * tau_hbar : tau_hbar, fco[k & 1], hiT(k), c, q, nq, sync);
  };
  const Rec* tw = reinterpret_cast<const Rec*>(p.Wln);
  if constexpr (SH::OWN) {
    Rec* own = tab + 2 * (SH::NHI + SH::NLO);
    for (int k = t; k < N / R; k += blockDim.x) own[k] = tw[k * R + (int)c];
    tw = own;
  }
  if constexpr (R > 1) {
    if (t < 6) {
      const uint32_t n = t < 2 ? R * SH::NW : R;  // arrivals: the cluster's warps, or its blocks
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"((uint32_t)__cvta_generic_to_shared(mb + t)), "r"(n)
                   : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    cluster_sync();  // every block is there, its mbarriers ready
  }
  __syncthreads();  // the step index is read
  const bool obs = !BATCH && p.obs;
  // The coefficients at the time of a record, in fco[m & 1]: those of the last potential phase,
  // or (a record of the state as it is, and after a kinetic half step) formed by the table warps
  // while the others load or finish.
  [[maybe_unused]] auto record_time = [&] { return p.g.t0 + (double)(s0 + m) * dt; };
  [[maybe_unused]] const bool coefs = obs && !(vkv && m > 0);
  static_assert(BATCH || SH::TW > 0, "");
  // One barrier of the block per phase: the tables of phase k are complete, and those of phase
  // k - 1 no longer read.
  if constexpr (SH::TW > 0) {
    if (t >= NT) {
      for (int64_t k = 0; k < nphase; k++) {
        make(k, t - NT, SH::TW, [] { asm volatile("bar.sync 2, %0;" ::"n"(SH::TW) : "memory"); });
        __syncthreads();
      }
      if (coefs) {
        record_coefs(*p.pot, record_time(), fco[m & 1], t - NT);
        __syncthreads();
      }
      __syncthreads();
      if constexpr (R > 1) cluster_sync();
      return;
    }
  }
  LN ln{s, red, cred, mb, p.ctrl, 0, t, c, 0u, 0u, false};
  V x[P];
  bool zero = false;
  int bad = 0;
  if constexpr (F::fixed_point) {
    cx<double> v[P];
#pragma unroll
    for (int k = 0; k < P; k++) v[k] = p.psi[ln.point(k)];
    auto top = [&] {
      uint32_t w = 0, none = 0;
#pragma unroll
      for (int k = 0; k < P; k++) w = max(w, max(fxp::whi(v[k].re) & 0x7fffffffu, fxp::whi(v[k].im) & 0x7fffffffu));
      ln.reduce(w, none, true);
      return w;
    };
    uint32_t mx = top();
    // all below 2^-953: off the denormals
    const bool tiny = mx < (70u << 20);
#pragma unroll
    for (int k = 0; k < P; k++)
      if (tiny) v[k] = mk(v[k].re * 0x1p900, v[k].im * 0x1p900);
    ln.bar();
    mx = top();
    zero = mx == 0u;
    bad = mx >= 0x7ff00000u;
    const uint32_t E = zero || bad ? 1023u : mx >> 20;
    ln.ex = (int32_t)E + 1 - (tiny ? 900 : 0);
    ln.bar();  // the reductions' words are free
#pragma unroll
    for (int k = 0; k < P; k++) {
      const uint32_t rh = fxp::whi(v[k].re), ih = fxp::whi(v[k].im);
      x[k] = mk(fx_from_double(rh, fxp::wlo(v[k].re), E + 1u - ((rh >> 20) & 0x7ffu)),
                fx_from_double(ih, fxp::wlo(v[k].im), E + 1u - ((ih >> 20) & 0x7ffu)));
    }
  } else {
#pragma unroll
    for (int k = 0; k < P; k++) x[k] = p.psi[ln.point(k)];
  }
  const bool stat = p.static_mask != 0, plane = p.plane_mask != 0;
  [[maybe_unused]] Rec Sk[SH::KEEP ? P : 1], Kk[SH::KEEP ? P : 1];
  if constexpr (SH::KEEP) {
#pragma unroll
    for (int k = 0; k < P; k++) {
      Kk[k] = F::kinetic(p, 0)[ln.point(k)];
      if (stat) Sk[k] = F::statics(p, 0)[ln.point(k)];
    }
  }
  auto potential = [&](int64_t kph) {
    if constexpr (SH::TW == 0) {
      ln.bar();
      make(kph, t, NT, [] { LN::bar(); });
    }
    __syncthreads();
    const Rec* hi = hiT(kph);
    const Rec* lo = hi + SH::NHI;
    const double* fc = fco[kph & 1];
    const bool half = phase_half(kph);
    const double tau = half ? 0.5 * dt : dt, tm0 = phase_time(kph);
    const Rec* S = F::statics(p, half ? 1 : 0);
    const DevPot& pot = *p.pot;
#pragma unroll
    for (int k = 0; k < P; k++) {
      const int i = ln.point(k);
      if (stat) {
        Rec w;
        if (SH::KEEP && !half)
          w = Sk[SH::KEEP ? k : 0];
        else
          w = S[i];
        bad |= F::bad(w);
        x[k] = F::mul(x[k], w);
      }
      if (plane) {
        x[k] = F::mul(x[k], hi[i >> SH::LOGLO]);
        x[k] = F::mul(x[k], lo[i & (SH::NLO - 1)]);
      }
    }
    if (plane) bad |= F::bad(hi[t % SH::NHI]) | F::bad(lo[ln.point(0) & (SH::NLO - 1)]);
    if (p.gen_mask) {
      // a loop, its body being long FP64 code; x rotates, so that nothing indexes registers
#pragma unroll 1
      for (int k = 0; k < P; k++) {
        const double xi = p.g.xmin[0] + (double)ln.point(k) * p.g.dx[0];
        double W = 0.0;
        for (int e = 0; e < pot.nterms; e++) {
          if (!((p.gen_mask >> e) & 1u)) continue;
          const wp_pot_term& tm = pot.term[e];
          const double sh = (tm.shape == WP_SHAPE_GAUSS) ? gauss_axis_factor(tm, 0, xi, tm0) : term_axis_part(tm, 0, xi, tm0);
          W += fc[e] * sh;
        }
        double sn, cs;
        sincos(-W * tau / p.g.hbar, &sn, &cs);
        const Rec w = F::rec(cs, sn);
        bad |= F::bad(w);
        const V v = F::mul(x[0], w);
#pragma unroll
        for (int q = 0; q < P - 1; q++) x[q] = x[q + 1];
        x[P - 1] = v;
      }
    }
  };
  auto kinetic = [&](int half) {
    const Rec* K = F::kinetic(p, half);
    auto factor = [&](int k) {
      Rec w;
      if (SH::KEEP && !half)
        w = Kk[SH::KEEP ? k : 0];
      else
        w = K[ln.point(k)];
      bad |= F::bad(w);
      return F::mul(x[k], w);
    };
    if constexpr (F::fixed_point) {
      // forward, factor with the exchange for the inverse, inverse: one copy of the code
#pragma unroll 1
      for (int it = 0; it < 2; it++) {
        ln.template fft<false>(x, tw);
        if (it == 0) {
#pragma unroll
          for (int k = 0; k < P; k++) x[k] = swapped(factor(k));
        }
      }
#pragma unroll
      for (int k = 0; k < P; k++) x[k] = swapped(x[k]);
      ln.ex -= LOGN;  // 1/N
    } else {
      ln.template fft<false>(x, tw);
#pragma unroll
      for (int k = 0; k < P; k++) x[k] = factor(k);
      ln.template fft<true>(x, tw);
    }
  };
  // VKV: P K P .. K P; KVK: K P K .. P K. One call of each, so that their code is there once.
  if (m > 0) {
#pragma unroll 1
    for (int64_t k = 0; k <= m; k++) {
      if (vkv || k > 0) potential(vkv ? k : k - 1);
      if (!vkv || k < m) kinetic(!vkv && (k == 0 || k == m) ? 1 : 0);
    }
  }
  // A value that is not finite has spread over the line by the transforms of a step; in fixed
  // point it is a flag, which the line's threads share here.
  bool nan = false;
  if constexpr (F::fixed_point) {
    uint32_t b = (uint32_t)bad, none = 0;
    ln.bar();
    ln.reduce(b, none);
    nan = b != 0u;
  }
  [[maybe_unused]] const double qnan = __longlong_as_double(0x7ff8000000000000ll);
  [[maybe_unused]] const bool chk = ln.ex < 200 || ln.ex > 1900;
  auto value = [&](V v) {  // the stored form of a point
    if constexpr (F::fixed_point) {
      uint32_t rh, rl, ih, il;
      fx_to_double(v.re, ln.ex, rh, rl);
      fx_to_double(v.im, ln.ex, ih, il);
      cx<double> y = mk(__hiloint2double((int)rh, (int)rl), __hiloint2double((int)ih, (int)il));
      if (chk) y = fxp::scaled(v, ln.ex - 1085);
      if (zero) y = mk(0.0, 0.0);
      if (nan) y = mk(qnan, qnan);
      return y;
    } else {
      return v;
    }
  };
  // The linear and constant terms of a record, alpha + beta i at grid point i: from the sums of
  // x |psi|^2 and |psi|^2 they would cancel on a box far from the origin. The general terms
  // follow below.
  [[maybe_unused]] const DevPot& pot = *p.pot;
  [[maybe_unused]] const double tm0 = record_time();
  [[maybe_unused]] const double* fr = fco[m & 1];
  [[maybe_unused]] double alpha = 0.0, beta = 0.0;
  if (coefs) __syncthreads();
  if (obs) {
    for (int e = 0; e < pot.nterms; e++) {
      if (!((p.plane_mask >> e) & 1u)) continue;
      const wp_pot_term& tm = pot.term[e];
      if (tm.shape == WP_SHAPE_LINEAR) {
        const double fa = fr[e] * tm.a[0];
        beta = fma(fa, p.g.dx[0], beta);
        alpha = fma(fa, p.g.xmin[0] - (tm.c0[0] + tm.v[0] * tm0), alpha);
      } else {
        alpha += fr[e];
      }
    }
  }
  double acc[NQ];
#pragma unroll
  for (int q = 0; q < NQ; q++) acc[q] = 0.0;
#pragma unroll
  for (int k = 0; k < P; k++) {
    const int i = ln.point(k);
    cx<T> v = value(x[k]);
    if (R > 1 && ln.lost) v = mk(T(qnan), T(qnan));  // never taken for a result
    if (m > 0) p.psi[i] = v;
    if (obs) {
      const double re = to_f64(v.re), im = to_f64(v.im);
      const double rho = fma(re, re, im * im), xi = p.g.xmin[0] + (double)i * p.g.dx[0], xr = xi * rho;
      acc[Q_RHO] += rho;
      acc[Q_X] += xr;
      acc[Q_XX] += xi * xr;
      acc[Q_V] += (p.Vs[i] + fma(beta, (double)i, alpha)) * rho;
      if (p.autocorr) {
        const cx<T> z = p.psi0[i];
        const double zr = to_f64(z.re), zi = to_f64(z.im);
        acc[Q_AC_RE] += zr * re + zi * im;
        acc[Q_AC_IM] += zr * im - zi * re;
      }
    }
  }
  if (obs) {
    if (p.gen_mask) {
#pragma unroll 1
      for (int k = 0; k < P; k++) {
        const double xi = p.g.xmin[0] + (double)ln.point(k) * p.g.dx[0];
        const cx<T> v = value(x[0]);
        const double re = to_f64(v.re), im = to_f64(v.im);
        double W = 0.0;
        for (int e = 0; e < pot.nterms; e++) {
          if (!((p.gen_mask >> e) & 1u)) continue;
          const wp_pot_term& tm = pot.term[e];
          W += fr[e] * ((tm.shape == WP_SHAPE_GAUSS) ? gauss_axis_factor(tm, 0, xi, tm0) : term_axis_part(tm, 0, xi, tm0));
        }
        acc[Q_V] += W * fma(re, re, im * im);
        const V first = x[0];
#pragma unroll
        for (int q = 0; q < P - 1; q++) x[q] = x[q + 1];
        x[P - 1] = first;
      }
    }
    const uint32_t ac = p.autocorr ? 3u << Q_AC_RE : 0u;
    total(ln, acc, ac | (1u << Q_RHO) | (1u << Q_X) | (1u << Q_XX) | (1u << Q_V), redd, part[0], 0, qp);
    ln.template fft<false>(x, tw);
#pragma unroll
    for (int q = 0; q < NQ; q++) acc[q] = 0.0;
#pragma unroll
    for (int k = 0; k < P; k++) {
      const cx<T> v = value(x[k]);
      const double re = to_f64(v.re), im = to_f64(v.im);
      const double rho = fma(re, re, im * im), kk = wavenumber(p.g, 0, ln.point(k)), kr = kk * rho;
      acc[Q_RHOK] += rho;
      acc[Q_K] += kr;
      acc[Q_K2] += kk * kr;
    }
    total(ln, acc, (1u << Q_RHOK) | (1u << Q_K) | (1u << Q_K2), redd, part[1], 1, qm);
    if (t < 32 && c == 0u) publish_obs(qp, qm, p.g, p.autocorr, tm0, s0 + m, t, p.ctrl, p.obs_out, p.obs_cap);
  }
  if (t == 0 && c == 0u) p.ctrl->step = s0 + m;
  if constexpr (SH::TW > 0) __syncthreads();
  if constexpr (R > 1) cluster_sync();  // no block leaves while another may write to it
}

template <class T, int LOGN, int LOGR>
__global__ void __launch_bounds__(Shape<T, LOGN, LOGR>::NT + Shape<T, LOGN, LOGR>::TW)
    k_line(const Res1dParams<T> p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  pass_begin();
  body<T, LOGN, LOGR, false>(p, smem_raw);
}

// Cluster b runs instance b (all of one line length) for nsteps.
template <class T, int LOGN, int LOGR>
__global__ void __launch_bounds__(Shape<T, LOGN, LOGR, true>::NT + Shape<T, LOGN, LOGR, true>::TW,
                                  Shape<T, LOGN, LOGR, true>::MIN_BLOCKS)
    k_line_batch(const Res1dParams<T>* __restrict__ params, int64_t nsteps) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(16) unsigned char raw[sizeof(Res1dParams<T>)];
  Res1dParams<T>& p = *reinterpret_cast<Res1dParams<T>*>(raw);
  const int* src = reinterpret_cast<const int*>(&params[blockIdx.x >> LOGR]);
  for (int k = threadIdx.x; k < (int)(sizeof(Res1dParams<T>) / sizeof(int)); k += blockDim.x)
    reinterpret_cast<int*>(raw)[k] = src[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    p.nsteps = nsteps;
    p.obs = 0;
  }
  __syncthreads();
  body<T, LOGN, LOGR, true>(p, smem_raw);
}

}  // namespace line
}  // namespace wp
