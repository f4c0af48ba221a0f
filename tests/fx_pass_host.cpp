// Host build of wp_fx.h in the two forms that the device kernels take a line through it: the
// passes' (wp_fx_pass.cuh: the bound of the inputs for the whole transform, sums in units of
// 2^kFxPassSum) and the resident lines' (wp_line.cuh: a second bound after 64 points from
// 2048 points on, sums in units of 2^kFxLineSum). Reads a command word, log2 n and n complex
// doubles from stdin (binary), writes n complex doubles to stdout:
//   0 a pass: load from doubles, forward transform
//   1 two passes: forward transform, the line stored in fixed point and loaded again,
//     inverse transform (n times the input)
//   2 a resident line: forward transform
//   3 the line's integers as loaded from doubles, stored in fixed point and read point by point
#define __host__
#define __device__
#define __forceinline__ inline
#include <algorithm>
#include <cstdio>
#include <vector>

#include "wp_fx.h"

using namespace wp;
using C = cx<int64_t>;

static void words(double x, uint32_t& hi, uint32_t& lo) {
  uint64_t b;
  memcpy(&b, &x, 8);
  hi = (uint32_t)(b >> 32);
  lo = (uint32_t)b;
}
static uint32_t absh(int64_t v) { return (uint32_t)(v >> 32) ^ (uint32_t)(v >> 63); }
static int64_t shift_jam(int64_t v, int32_t k) { return k < 0 ? (int64_t)((uint64_t)v << -k) : ((v >> k) | 1); }
static int64_t load(double x, uint32_t E2) {
  uint32_t hi, lo;
  words(x, hi, lo);
  return fx_from_double(hi, lo, E2 - ((hi >> 20) & 0x7ffu));
}

// A line in fixed point: an integer x stands for x 2^(ex - 1085).
template <int LOGN>
struct Line {
  static constexpr int N = 1 << LOGN;
  std::vector<C> x = std::vector<C>(N);
  int32_t ex = 0;
  FxSchedule sc;
  int32_t bS = 0;

  // stages from span 2^LS0 to 2^LS1 under sc
  void stages(int ls0, int ls1) {
    const long double pi = 3.141592653589793238462643383279502884L;
    std::vector<C> y(N);
    int t = 0;
    for (int ls = ls0; ls < ls1; t++) {
      const int lr = wp_stage_radix_log(LOGN, ls), R = 1 << lr, nr = N >> lr, ns = 1 << ls;
      for (int j = 0; j < nr; j++) {
        C v[8];
        const int jm = j & (ns - 1);
        for (int r = 0; r < R; r++) {
          v[r] = x[j + r * nr];
          if (ls == 0) continue;
          const long double a = -2.0L * pi * (long double)(r * jm) / (long double)(ns * R);
          if (r == 0)
            v[r] = {v[r].re >> (2 - sc.at[t]), v[r].im >> (2 - sc.at[t])};
          else
            v[r] = fx_cmul(v[r], fx_rec_host(cosl(a), sinl(a)), sc.at[t]);
        }
        R == 8 ? fx_dft<8>(v) : fx_dft<4>(v);
        const int d0 = ((j >> ls) << (ls + lr)) + jm;
        for (int r = 0; r < R; r++) y[d0 + (r << ls)] = v[r];
      }
      x.swap(y);
      ls += lr;
    }
  }
  uint32_t largest() const {
    uint32_t any = 0;
    for (const C& v : x) any |= absh(v.re) | absh(v.im);
    return any;
  }
  // a pass's bounds of doubles, the integers and the transform
  void pass(const std::vector<double>& d) {
    uint32_t m = 0, L = 0, hi, lo;
    for (double v : d) {
      words(v, hi, lo);
      m = std::max(m, hi & 0x7fffffffu);
    }
    const uint32_t E = m >> 20;
    for (double v : d) {
      words(v, hi, lo);
      L += fx_mag<kFxPassSum>(hi, E - ((hi >> 20) & 0x7ffu));
    }
    sc = fx_schedule<LOGN>(64, fx_sum_bits<kFxPassSum>(L));
    const uint32_t E2 = E + (uint32_t)sc.first;
    ex = (int32_t)E2;
    for (int i = 0; i < N; i++) x[i] = {load(d[2 * i], E2), load(d[2 * i + 1], E2)};
    stages(0, LOGN);
    ex += sc.total - sc.first;
  }
  // the points as the passes store them between them: re lo, re hi, im lo, im hi
  std::vector<uint32_t> stored() const {
    std::vector<uint32_t> w(4 * N);
    for (int i = 0; i < N; i++) {
      const int up = std::max(fx_clz(absh(x[i].re) | absh(x[i].im)) - 1, 0);
      const uint32_t code = (uint32_t)(ex - up + kFxBias);
      const uint64_t re = (uint64_t)x[i].re << up, im = (uint64_t)x[i].im << up;
      w[4 * i] = ((uint32_t)re & ~63u) | (code >> 6);
      w[4 * i + 1] = (uint32_t)(re >> 32);
      w[4 * i + 2] = ((uint32_t)im & ~63u) | (code & 63u);
      w[4 * i + 3] = (uint32_t)(im >> 32);
    }
    return w;
  }
  // loaded again with its new bounds, transformed
  void store_and_pass() {
    const std::vector<uint32_t> w = stored();
    auto mag = [](uint32_t h) { return h ^ (uint32_t)((int32_t)h >> 31); };
    uint32_t m = 0, L = 0;
    for (int i = 0; i < N; i++) m = std::max(m, fx_code(w[4 * i], w[4 * i + 2]));
    for (int i = 0; i < N; i++) {
      const uint32_t s = m - fx_code(w[4 * i], w[4 * i + 2]);
      L += fx_mag_int<kFxPassSum>(fx_shr64(mag(w[4 * i + 1]), 0u, s)) + fx_mag_int<kFxPassSum>(fx_shr64(mag(w[4 * i + 3]), 0u, s));
    }
    sc = fx_schedule<LOGN>(64, fx_sum_bits<kFxPassSum>(L));
    ex = (int32_t)m - kFxBias + sc.first;
    const uint32_t right = sc.first > 0 ? (uint32_t)sc.first : 0u, left = sc.first < 0 ? (uint32_t)-sc.first : 0u;
    for (int i = 0; i < N; i++) {
      const uint32_t s = m - fx_code(w[4 * i], w[4 * i + 2]) + right;
      x[i] = {(int64_t)((uint64_t)fx_align(w[4 * i], (int32_t)w[4 * i + 1], s) << left),
              (int64_t)((uint64_t)fx_align(w[4 * i + 2], (int32_t)w[4 * i + 3], s) << left)};
    }
    for (C& v : x) v = {v.im, v.re};
    stages(0, LOGN);
    for (C& v : x) v = {v.im, v.re};
    ex += sc.total - sc.first;
  }
  // a resident line's
  void resident(const std::vector<double>& d) {
    uint32_t m = 0, hi, lo;
    for (double v : d) {
      words(v, hi, lo);
      m = std::max(m, hi & 0x7fffffffu);
    }
    const uint32_t E2 = (m >> 20) + 1u;
    ex = (int32_t)E2;
    uint32_t L = 0;
    for (int i = 0; i < N; i++) {
      x[i] = {load(d[2 * i], E2), load(d[2 * i + 1], E2)};
      L += fx_mag_int<kFxLineSum>(absh(x[i].re)) + fx_mag_int<kFxLineSum>(absh(x[i].im));
    }
    bS = fx_sum_bits<kFxLineSum>(L);
    constexpr bool mid = fx_mid(LOGN);
    sc = fx_schedule<LOGN, 0, mid ? kFxMidLog : LOGN>(65 - fx_clz(largest()), bS);
    scale();
    stages(0, mid ? kFxMidLog : LOGN);
    if (mid) {
      sc = fx_schedule<LOGN, mid ? kFxMidLog : 0, LOGN>(65 - fx_clz(largest()), bS);
      scale();
      stages(kFxMidLog, LOGN);
    }
  }
  // the integers of doubles at the line's exponent, stored and read back each by itself
  void points(std::vector<double>& d) {
    uint32_t m = 0, hi, lo;
    for (double v : d) {
      words(v, hi, lo);
      m = std::max(m, hi & 0x7fffffffu);
    }
    ex = (int32_t)(m >> 20);
    for (int i = 0; i < N; i++) x[i] = {load(d[2 * i], (uint32_t)ex), load(d[2 * i + 1], (uint32_t)ex)};
    const std::vector<uint32_t> w = stored();
    for (int i = 0; i < N; i++) {
      const int32_t e = (int32_t)fx_code(w[4 * i], w[4 * i + 2]) - kFxBias;
      for (int k = 0; k < 2; k++) {
        const int64_t v = fx_align(w[4 * i + 2 * k], (int32_t)w[4 * i + 2 * k + 1], 0);
        d[2 * i + k] = std::ldexp((double)v, e - 1085);
      }
    }
  }
  void scale() {
    ex += sc.total;
    bS -= sc.total;
    for (C& v : x) v = {shift_jam(v.re, sc.first), shift_jam(v.im, sc.first)};
  }
  void out(std::vector<double>& d) const {
    for (int i = 0; i < 2 * N; i++) {
      uint32_t hi, lo;
      fx_to_double(i & 1 ? x[i / 2].im : x[i / 2].re, ex, hi, lo);
      const uint64_t b = ((uint64_t)hi << 32) | lo;
      memcpy(&d[i], &b, 8);
    }
  }
};

template <int LOGN>
static int go(int cmd, std::vector<double>& d) {
  Line<LOGN> l;
  if (cmd == 3) {
    l.points(d);
    return 0;
  }
  if (cmd == 2) {
    l.resident(d);
  } else {
    l.pass(d);
    if (cmd == 1) l.store_and_pass();
  }
  l.out(d);
  return 0;
}

int main() {
  int32_t hdr[2];
  if (fread(hdr, sizeof(hdr), 1, stdin) != 1) return 2;
  if (hdr[0] < 0 || hdr[0] > 3 || hdr[1] < 5 || hdr[1] > 13) return 2;
  std::vector<double> d(2 << hdr[1]);
  if (fread(d.data(), 8, d.size(), stdin) != d.size()) return 2;
  switch (hdr[1]) {
    case 5: go<5>(hdr[0], d); break;
    case 6: go<6>(hdr[0], d); break;
    case 7: go<7>(hdr[0], d); break;
    case 8: go<8>(hdr[0], d); break;
    case 9: go<9>(hdr[0], d); break;
    case 10: go<10>(hdr[0], d); break;
    case 11: go<11>(hdr[0], d); break;
    case 12: go<12>(hdr[0], d); break;
    case 13: go<13>(hdr[0], d); break;
  }
  fwrite(d.data(), 8, d.size(), stdout);
  return 0;
}
