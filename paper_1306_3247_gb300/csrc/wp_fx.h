// 64-bit fixed-point arithmetic of the complex128 transforms (the Fourier transforms of
// eq. (ft), Sec. 2.1 of arXiv:1306.3247).
//
// GB300 issues one FP64 warp instruction per SM every 19 clocks (measured: 304 clocks for
// 16 warps, whatever the number of active lanes or independent chains) against four 32-bit
// integer ones per clock, so a complex128 pass written in FP64 is bound by that pipe: a
// 256-point transform is about 20 FP64 instructions per point, 1500 issue slots' worth.
// Between the load and the store of a pass a line is therefore held as 64-bit integers with
// one common exponent per line. A sum is exact and costs about 3.4 issue slots, a product
// with a unit factor about 60 (measured on GB300, 32-bit multiplies and high words).
//
// Accuracy. With M the largest |x| of a line and S its sum of |re| + |im|,
// every value a transform forms from q of its points is at most min(q M, S). The
// integers are scaled stage by stage so that this bound stays below 2^62 (fx_schedule):
// nothing overflows, and no bits are kept back for growth that a line cannot have. The few
// roundings (one when a double becomes an integer, one per product) are a small number of
// units, 2^-62 min(q M, S). For a line of m comparable points the bound is at most sqrt(q)
// times its 2-norm, so the transform's own rounding is a few 1e-17 relative in 2-norm for
// localised and for flat lines alike, below the 1e-16 of a value's FP64 rounding when the
// pass stores it.
//
// The functions compile for the device and, with WP_HD empty, as plain C++ for the CPU
// tests.
#pragma once

#include <cmath>
#include <cstdint>
#include <cstring>

#include "wp_internal.h"

#ifndef WP_HD
#define WP_HD __host__ __device__ __forceinline__
#endif

namespace wp {

WP_HD int32_t fx_mulhi(int32_t a, int32_t b) {
#ifdef __CUDA_ARCH__
  return __mulhi(a, b);
#else
  return (int32_t)(((int64_t)a * (int64_t)b) >> 32);
#endif
}
WP_HD uint32_t fx_shr64(uint32_t lo, uint32_t hi, uint32_t s) {  // low word of (hi:lo) >> min(s, 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_rc(lo, hi, s);
#else
  const uint64_t v = ((uint64_t)hi << 32) | lo;
  return (uint32_t)(v >> (s > 32 ? 32 : s));
#endif
}
WP_HD uint32_t fx_shl64(uint32_t lo, uint32_t hi, uint32_t s) {  // high word of (hi:lo) << min(s, 32)
#ifdef __CUDA_ARCH__
  return __funnelshift_lc(lo, hi, s);
#else
  const uint64_t v = ((uint64_t)hi << 32) | lo;
  return s >= 32 ? lo : (uint32_t)((v << s) >> 32);
#endif
}
WP_HD int fx_clz(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __clz((int)v);
#else
  return v ? __builtin_clz(v) : 32;
#endif
}

// v = h 2^32 + l with a signed low half.
struct FxHalves {
  int32_t h, l;
};
WP_HD FxHalves fx_halves(int64_t v) {
  FxHalves r;
  r.l = (int32_t)v;
  r.h = (int32_t)(v >> 32) + (int32_t)((uint32_t)r.l >> 31);
  return r;
}
// x c / 2^64: the high product and the floors of the two cross products (the low product is
// below a quarter of a unit), on average one unit low. Products are used in differences, where
// that cancels; a zero stays zero.
WP_HD int64_t fx_mul(FxHalves x, int32_t ch, int32_t cl) {
  const uint32_t lo = (uint32_t)x.h * (uint32_t)ch;
  const int64_t hh = (int64_t)(((uint64_t)(uint32_t)fx_mulhi(x.h, ch) << 32) | lo);
  return hh + (int64_t)(fx_mulhi(x.h, cl) + fx_mulhi(x.l, ch));
}

// Unit factor c + i s: c, c + s and c - s times 2^62, split into halves. A low half that is
// zero becomes -1 (2^-62 off): a product's floor would be exact with it, and no longer cancel
// against another's.
WP_HD FxRec fx_rec(int64_t c, int64_t s) {
  FxRec r;
  const FxHalves a = fx_halves(c), b = fx_halves(c + s), d = fx_halves(c - s);
  r.ch = a.h, r.cl = a.l ? a.l : -1;
  r.ph = b.h, r.pl = b.l ? b.l : -1;
  r.mh = d.h, r.ml = d.l ? d.l : -1;
  r.bad = r.reserved = 0;
  return r;
}

// v (c + i s) 2^(sh - 2) in three products: with t = c (re + im), re c - im s =
// t - im (c + s) and im c + re s = t - re (c - s).
WP_HD cx<int64_t> fx_cmul(cx<int64_t> v, const FxRec& w, uint32_t sh = 2) {
  const FxHalves x = fx_halves(v.re), y = fx_halves(v.im), z = fx_halves(v.re + v.im);
  const int64_t t = fx_mul(z, w.ch, w.cl);
  cx<int64_t> r;
  r.re = (int64_t)((uint64_t)(t - fx_mul(y, w.ph, w.pl)) << sh);
  r.im = (int64_t)((uint64_t)(t - fx_mul(x, w.mh, w.ml)) << sh);
  return r;
}

// Scaling of the stages of a 2^LOGN-point transform (stage plan wp_stage_radix_log) from span
// 2^LS0 to 2^LS1: |inputs| < 2^bM, line sums of the transform's inputs < 2^bS. first: the
// right shift of the inputs (negative: left), at[t] = the shift that goes with the twiddles
// of the t-th of these stages (fx_cmul; a point without a twiddle shifts right by
// 2 - at[t]; the stage at span 1 has none), total: the whole right shift. A stage shifts by
// at most two bits, which the products take for free: where the bound grows by three, the
// stages before run one bit lower.
struct FxSchedule {
  int32_t first, total;
  uint32_t at[4];
};
template <int LOGN, int LS0 = 0, int LS1 = LOGN>
WP_HD FxSchedule fx_schedule(int32_t bM, int32_t bS) {
  FxSchedule r;
  // B[t]: bits before stage t; B[0] those of the inputs, or with no twiddles to shift at the
  // first stage those after it
  int32_t B[6] = {0, 0, 0, 0, 0, 0};
  int ns = 0;
  B[0] = bM < bS ? bM : bS;
#pragma unroll
  for (int ls = LS0; ls < LS1;) {
    ls += wp_stage_radix_log(LOGN, ls);
    const int32_t b = bM + ls - LS0;
    B[++ns] = b < bS ? b : bS;
  }
  if (LS0 == 0) B[0] = B[1];
#pragma unroll
  for (int t = 4; t >= 0; t--)
    if (t < ns && B[t] < B[t + 1] - 2) B[t] = B[t + 1] - 2;
  if (LS0 == 0) B[0] = B[1];
  r.first = B[0] - 62;
#pragma unroll
  for (int t = 0; t < 4; t++) r.at[t] = t < ns ? (uint32_t)(2 - (B[t + 1] - B[t])) : 2u;
  r.total = B[ns] - 62;
  return r;
}
// Resident lines of 2^11 points and more take their bound anew after 64 points (span 2^6): the
// line sum alone is far above the values that a long line of many comparable points forms.
// Passes take the bound of their inputs through to the end.
constexpr int kFxMidLog = 6;
WP_HD constexpr bool fx_mid(int logn) { return logn >= 11; }

// x / sqrt(2): the constant times 2^63; one cross product rounded down, the other up.
WP_HD int64_t fx_rsqrt2(int64_t x) {
  constexpr int64_t c = 6521908912666391106ll;
  constexpr int32_t ch = (int32_t)((c + 0x80000000ll) >> 32), cl = (int32_t)c;
  const FxHalves v = fx_halves(x);
  const uint32_t lo = (uint32_t)v.h * (uint32_t)ch;
  const int64_t hh = (int64_t)(((uint64_t)(uint32_t)fx_mulhi(v.h, ch) << 32) | lo);
  return (int64_t)((uint64_t)(hh + (int64_t)(fx_mulhi(v.h, cl) - fx_mulhi(v.l, -ch))) << 1);
}

// Forward DFT of R = 4 or 8 points in place, natural order in and out.
WP_HD void fx_dft4(cx<int64_t>& x0, cx<int64_t>& x1, cx<int64_t>& x2, cx<int64_t>& x3) {
  const cx<int64_t> a0 = {x0.re + x2.re, x0.im + x2.im}, a1 = {x0.re - x2.re, x0.im - x2.im};
  const cx<int64_t> a2 = {x1.re + x3.re, x1.im + x3.im}, a3 = {x1.im - x3.im, x3.re - x1.re};  // -i (x1 - x3)
  x0 = {a0.re + a2.re, a0.im + a2.im};
  x2 = {a0.re - a2.re, a0.im - a2.im};
  x1 = {a1.re + a3.re, a1.im + a3.im};
  x3 = {a1.re - a3.re, a1.im - a3.im};
}
template <int R>
WP_HD void fx_dft(cx<int64_t>* v) {
  if (R == 4) {
    fx_dft4(v[0], v[1], v[2], v[3]);
  } else {
    // DFTs of the even and odd halves, combined with the powers of exp(-2 pi i / 8)
    fx_dft4(v[0], v[2], v[4], v[6]);
    fx_dft4(v[1], v[3], v[5], v[7]);
    const cx<int64_t> o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7], e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    const cx<int64_t> t1 = {fx_rsqrt2(o1.re + o1.im), fx_rsqrt2(o1.im - o1.re)};
    const cx<int64_t> t3 = {fx_rsqrt2(o3.im - o3.re), fx_rsqrt2(o3.re + o3.im)};  // its imaginary part negated
    v[0] = {e0.re + o0.re, e0.im + o0.im};
    v[4] = {e0.re - o0.re, e0.im - o0.im};
    v[1] = {e1.re + t1.re, e1.im + t1.im};
    v[5] = {e1.re - t1.re, e1.im - t1.im};
    v[2] = {e2.re + o2.im, e2.im - o2.re};
    v[6] = {e2.re - o2.im, e2.im + o2.re};
    v[3] = {e3.re + t3.re, e3.im - t3.im};
    v[7] = {e3.re - t3.re, e3.im + t3.im};
  }
}

// Units of the 32-bit sums of |re| + |im| of a line, 2^UNIT. A part is below 2^63 and its
// magnitude rounded up at most 2^(63 - UNIT) units, so a line of n points sums to at most
// n 2^(64 - UNIT): below 2^32 for the 2048 points of a pass in units of 2^44 (in units of 2^43
// a flat line just below a power of two is 2^32 and its sum 0), and for the 8192 of a resident
// line in units of 2^46.
constexpr int kFxPassSum = 44, kFxLineSum = 46;

// |x| / 2^UNIT rounded up, of a double with high word hi and its leading one at bit 62 - s.
template <int UNIT = 43>
WP_HD uint32_t fx_mag(uint32_t hi, uint32_t s) {
  return fx_shr64(((hi & 0x000fffffu) | 0x00100000u) >> (UNIT - 42), 0u, s) + 1u;
}
// |x| / 2^UNIT rounded up, of an integer x with high word a of its magnitude rounded down.
template <int UNIT>
WP_HD uint32_t fx_mag_int(uint32_t a) {
  return (a >> (UNIT - 32)) + 1u;
}
// Bits of a line sum in units of 2^UNIT.
template <int UNIT = 43>
WP_HD int32_t fx_sum_bits(uint32_t L) {
  return 32 + UNIT - fx_clz(L);
}

// The double with words (hi, lo), its leading one moved to bit 62 - s. The last bit is set,
// which makes the error of the dropped bits symmetric (a plain floor would leave half a unit
// of the same sign on every point). Zero for s >= 64; a zero or denormal double, which has
// no leading one, needs such an s.
WP_HD int64_t fx_from_double(uint32_t hi, uint32_t lo, uint32_t s) {
  uint32_t mh = (hi & 0x000fffffu) | 0x00100000u;
  mh = (mh << 10) | (lo >> 22);
  uint32_t ml = lo << 10;
  const bool far = s >= 32u, none = s >= 64u;
  ml = far ? mh : ml;
  mh = far ? 0u : mh;
  s = far ? s - 32u : s;
  const uint32_t sg = none ? 0u : (uint32_t)((int32_t)hi >> 31);
  const uint32_t l = (fx_shr64(ml, mh, s) ^ sg) | (none ? 0u : 1u), h = fx_shr64(mh, 0u, s) ^ sg;
  return (int64_t)(((uint64_t)h << 32) | l);
}

// The double v 2^(e - 1085), rounded to nearest (ties away), where it is a normal number: e +
// 1 is the biased exponent of a value with the top bit 2^63 set.
WP_HD void fx_to_double(int64_t v, int32_t e, uint32_t& hi, uint32_t& lo) {
  const int64_t sg = v >> 63;
  const uint64_t m = (uint64_t)((v ^ sg) - sg);
  uint32_t h = (uint32_t)(m >> 32), l = (uint32_t)m;
  const bool low = h == 0u;
  h = low ? l : h;
  l = low ? 0u : l;
  const uint32_t k = (uint32_t)fx_clz(h);
  e -= (int32_t)k + (low ? 32 : 0);
  h = fx_shl64(l, h, k);
  l = l << (k & 31u);  // k = 32 only for v = 0
  // the leading one is bit 52 of (h:l) >> 11 and adds one to the exponent field, as does a
  // carry out of the rounding
  uint64_t b = ((((uint64_t)h << 32) | l) >> 11) + ((l >> 10) & 1u);
  b += (uint64_t)(uint32_t)(e << 20) << 32;
  if (h == 0u) b = 0;
  hi = (uint32_t)(b >> 32) | ((uint32_t)(sg >> 32) & 0x80000000u);
  lo = (uint32_t)b;
}

// Fixed-point points in memory, between the passes of a step: v x 2^(ex - 1085) with the low
// six bits of each part giving way to half of the exponent code ex + kFxBias. Code 0 is a
// point below the range, kFxNan one that is not finite.
constexpr int32_t kFxBias = 1200, kFxNan = 4095;
WP_HD uint32_t fx_code(uint32_t re_lo, uint32_t im_lo) { return ((re_lo & 63u) << 6) | (im_lo & 63u); }
// v >> s with the six code bits replaced by their middle and the last bit set (jam = 0: left
// as it is, so that a zero far below the line's largest stays zero).
WP_HD int64_t fx_align(uint32_t lo, int32_t hi, uint32_t s, uint32_t jam = 1u) {
  const bool far = s >= 32u;
  uint32_t l = (lo & ~63u) | 32u;
  const int32_t sg = hi >> 31;
  l = far ? (uint32_t)hi : l;
  const int32_t h = far ? sg : hi;
  s = far ? s - 32u : s;
  const uint32_t r = fx_shr64(l, (uint32_t)h, s) | jam;
  return (int64_t)(((uint64_t)(uint32_t)(h >> (s > 31u ? 31u : s)) << 32) | r);
}

// Host: a unit factor from its extended-precision value.
inline FxRec fx_rec_host(long double c, long double s) {
  const long double q = 4611686018427387904.0L;  // 2^62
  const bool ok = std::isfinite(c) && std::isfinite(s);
  FxRec r = ok ? fx_rec((int64_t)llroundl(c * q), (int64_t)llroundl(s * q)) : fx_rec(0, 0);
  r.bad = !ok;
  return r;
}

}  // namespace wp
