// Host build of the fixed-point arithmetic of the complex128 transforms (wp_fx.h), driven
// as the device passes drive it: bounds and scaling of a line, conversion from doubles, the
// Stockham stages with their schedule, conversion back. Reads a command word and its data
// from stdin (binary), writes doubles to stdout:
//   0 logn, 2^logn complex doubles -> the forward transform
//   1 n, n pairs of doubles (c, s) and n complex doubles v -> v (c + i s)
//   2 n, n complex doubles -> the same through the stored fixed-point form
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
static double value(int64_t v, int32_t ex) {
  uint32_t hi, lo;
  fx_to_double(v, ex, hi, lo);
  const uint64_t b = ((uint64_t)hi << 32) | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
}
// The largest exponent of x, and its line sum at that exponent.
static uint32_t bounds(const std::vector<double>& x, uint32_t& L) {
  uint32_t m = 0, hi, lo;
  for (double v : x) {
    words(v, hi, lo);
    m = std::max(m, hi & 0x7fffffffu);
  }
  L = 0;
  for (double v : x) {
    words(v, hi, lo);
    L += (fx_mag(hi, (m >> 20) - ((hi >> 20) & 0x7ffu)) >> 3) + 1u;  // units of 2^46: n up to 2^13
  }
  return m >> 20;
}
static int64_t load(double x, uint32_t E2) {
  uint32_t hi, lo;
  words(x, hi, lo);
  return fx_from_double(hi, lo, E2 - ((hi >> 20) & 0x7ffu));
}

template <int LOGN>
static void transform(std::vector<double>& d) {
  const int n = 1 << LOGN;
  uint32_t L;
  const uint32_t E = bounds(d, L);
  constexpr bool mid = fx_mid(LOGN);
  constexpr int kMid = mid ? kFxMidLog : LOGN;
  int32_t bS = fx_sum_bits(L) + 3;
  FxSchedule sc = fx_schedule<LOGN, 0, kMid>(64, bS);
  bS -= sc.total;
  const uint32_t E2 = E + (uint32_t)sc.first;
  int32_t ex = (int32_t)E2 + sc.total - sc.first;
  std::vector<C> x(n), y(n);
  for (int i = 0; i < n; i++) x[i] = {load(d[2 * i], E2), load(d[2 * i + 1], E2)};
  const long double pi = 3.141592653589793238462643383279502884L;
  int t = 0;
  for (int ls = 0; ls < LOGN; t++) {
    const int lr = wp_stage_radix_log(LOGN, ls), R = 1 << lr, nr = n >> lr, ns = 1 << ls;
    if (mid && ls == kMid) {
      uint32_t any = 0;
      for (const C& v : x)
        any |= ((uint32_t)(v.re >> 32) ^ (uint32_t)(v.re >> 63)) | ((uint32_t)(v.im >> 32) ^ (uint32_t)(v.im >> 63));
      sc = fx_schedule<LOGN, mid ? kFxMidLog : 0, LOGN>(65 - fx_clz(any), bS);
      ex += sc.total;
      t = 0;
      auto shift = [&](int64_t v) {
        return sc.first < 0 ? (int64_t)((uint64_t)v << -sc.first) : ((v >> sc.first) | 1);
      };
      for (C& v : x) v = {shift(v.re), shift(v.im)};
    }
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
  for (int i = 0; i < n; i++) {
    d[2 * i] = value(x[i].re, ex);
    d[2 * i + 1] = value(x[i].im, ex);
  }
}

int main() {
  int32_t hdr[2];
  if (fread(hdr, sizeof(hdr), 1, stdin) != 1) return 2;
  const int n = hdr[0] == 0 ? 1 << hdr[1] : hdr[1];
  if (n < 1 || n > (1 << 20)) return 2;
  std::vector<double> w(hdr[0] == 1 ? 2 * n : 0), d(2 * n);
  if (!w.empty() && fread(w.data(), 8, w.size(), stdin) != w.size()) return 2;
  if (fread(d.data(), 8, d.size(), stdin) != d.size()) return 2;
  if (hdr[0] == 0) {
    switch (hdr[1]) {
      case 6: transform<6>(d); break;
      case 7: transform<7>(d); break;
      case 8: transform<8>(d); break;
      case 9: transform<9>(d); break;
      case 10: transform<10>(d); break;
      case 11: transform<11>(d); break;
      case 12: transform<12>(d); break;
      case 13: transform<13>(d); break;
      default: return 2;
    }
  } else {
    uint32_t L;
    const uint32_t E2 = bounds(d, L) + 2u;
    for (int i = 0; i < n; i++) {
      C v = {load(d[2 * i], E2), load(d[2 * i + 1], E2)};
      int32_t ex = (int32_t)E2;
      if (hdr[0] == 1) {
        v = fx_cmul(v, fx_rec_host(w[2 * i], w[2 * i + 1]));
      } else {
        // stored with its exponent code, read with an exponent distance of three
        const uint32_t code = (uint32_t)(ex + kFxBias);
        const uint32_t rl = ((uint32_t)v.re & ~63u) | (code >> 6), il = ((uint32_t)v.im & ~63u) | (code & 63u);
        if (fx_code(rl, il) != code) return 3;
        v = {fx_align(rl, (int32_t)(v.re >> 32), 3), fx_align(il, (int32_t)(v.im >> 32), 3)};
        ex = (int32_t)fx_code(rl, il) - kFxBias + 3;
      }
      d[2 * i] = value(v.re, ex);
      d[2 * i + 1] = value(v.im, ex);
    }
  }
  fwrite(d.data(), 8, d.size(), stdout);
  return 0;
}
