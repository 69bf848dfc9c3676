// The fixed-point reconstructions of ase_df_fixed.cuh compiled for the host, against exact weights in long
// double and beside the FP64 chains that they stand in for (lin_eval, lin_gauss_sym).
// exact_weights.h is written by test_fixed_point.py: per order the weights as doubles (as the tables
// hold them) and as long doubles.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

using std::max;
using std::min;
#define __device__
#define __constant__ static const
#define __forceinline__ inline
static inline long long __double_as_longlong(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline double __longlong_as_double(long long b) { double x; std::memcpy(&x, &b, 8); return x; }
static inline int __float_as_int(float x) { int b; std::memcpy(&b, &x, 4); return b; }
static inline float __uint2float_rz(unsigned w) {  // toward zero: the bits beyond 24 cut off
  int drop = 0;
  while (w >> drop >= 1u << 24) ++drop;
  return std::ldexp((float)(w >> drop), drop);
}
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (unsigned)((((uint64_t)hi << 32) | lo) << (s & 31u) >> 32);
}
#include "ase_df_fixed.cuh"
#include "exact_weights.h"

static std::mt19937_64 rng(20241009);
static double uni() { return (double)(rng() >> 11) * 0x1p-53; }
static long bad = 0;
static void fail(const char* what, int r, double a, double b) {
  if (bad++ < 10) std::printf("%s, order %d: %a %a\n", what, r, a, b);
}
static bool same(double a, double b) { return __double_as_longlong(a) == __double_as_longlong(b); }

// FP64 chains
static double lin(int r, const double* v, bool mirror, const Exact& X) {
  const int K = (r - 1) / 2;
  double s = X.f[mirror ? 2 * K : 0] * v[-K];
  for (int t = 1; t < r; ++t) s = std::fma(X.f[mirror ? 2 * K - t : t], v[t - K], s);
  return s;
}
static void gauss(int r, int G, const double* v, const Exact& X, double* out) {
  const int K = (r - 1) / 2;
  if (G == 1) {
    out[0] = std::fma(X.e[0][1], v[1], std::fma(X.e[0][0], v[0], X.e[0][1] * v[-1]));
    return;
  }
  for (int g = 0; g < (G + 1) / 2; ++g) {
    double E = X.e[g][0] * v[0], O = 0.0;
    for (int t = 1; t <= K; ++t) E = std::fma(X.e[g][t], v[t] + v[-t], E);
    for (int t = 1; t <= K; ++t) O = t == 1 ? X.o[g][1] * (v[1] - v[-1]) : std::fma(X.o[g][t], v[t] - v[-t], O);
    out[g] = 2 * g + 1 == G ? E : E + O;
    if (2 * g + 1 < G) out[G - 1 - g] = E - O;
  }
}

// what a pattern's stencil holds, in units of its largest value
enum { SMOOTH, NOISE, TAIL, SPREAD, PATTERNS };
static const char* kName[] = {"smooth", "noise", "one large value", "spread over the range"};
static void draw(int pattern, int n, double* v) {
  const double a = 0.2 * uni(), k = uni(), p = 6.3 * uni();
  const int big = (int)(rng() % n);
  for (int t = 0; t < n; ++t) {
    const double x = 1.0 + uni();
    switch (pattern) {
      case SMOOTH: v[t] = 1.5 * (1.0 + a * std::sin(k * t + p)); break;
      case NOISE: v[t] = x; break;
      case TAIL: v[t] = t == big ? x : std::ldexp(x, -asedf::kFixRange); break;
      default: v[t] = std::ldexp(x, -(int)(rng() % (asedf::kFixRange + 1)));
    }
  }
}

template <int R>
static void check(const Exact& X) {
  constexpr int K = (R - 1) / 2, G = R == 3 ? 1 : K;
  double buf[3 * R], rev[R], neg[R], out[2], o2[2], g1[4], g2[4];
  double* v = buf + K;
  // constants, over all exponents served: the same bits
  for (int i = 0; i < 20000; ++i) {
    const double c = std::ldexp((rng() & 1 ? 1.0 : -1.0) * (1.0 + uni()), (int)(rng() % 1199) - 959);
    for (int t = 0; t < R; ++t) buf[t] = c;
    if (!asedf::fix_normal<R, 2>(v, 1, out) || !same(out[0], c) || !same(out[1], c)) fail("constant", R, out[0], c);
    if (!asedf::fix_gauss<R, G>(v, 1, g1)) fail("constant refused", R, c, c);
    for (int q = 0; q < G; ++q)
      if (!same(g1[q], c)) fail("constant at a Gauss point", R, g1[q], c);
  }
  // zeros, and what has to be refused
  for (int t = 0; t < R; ++t) buf[t] = t & 1 ? -0.0 : 0.0;
  if (!asedf::fix_normal<R, 2>(v, 1, out) || !same(out[0], 0.0) || !same(out[1], 0.0)) fail("zeros", R, out[0], out[1]);
  if (!asedf::fix_gauss<R, G>(v, 1, g1) || !same(g1[0], 0.0)) fail("zeros at a Gauss point", R, g1[0], 0.0);
  for (int t = 0; t < R; ++t)
    for (const double x : {0.0, -1.0, 1.0 / 0.0, -1.0 / 0.0, 0.0 / 0.0, 0x1p-1074, -std::ldexp(1.9, -asedf::kFixRange - 1),
                           std::ldexp(1.0, asedf::kFixRange + 1), 1e300}) {
      for (int k = 0; k < R; ++k) buf[k] = 1.0;
      buf[t] = x;
      if (asedf::fix_normal<R, 2>(v, 1, out) || asedf::fix_gauss<R, G>(v, 1, g1)) fail("not refused", R, x, t);
    }
  for (const double x : {0x1p241, 0x1p-960, 0x1p-1074}) {
    for (int k = 0; k < R; ++k) buf[k] = x;
    if (asedf::fix_normal<R, 2>(v, 1, out)) fail("exponent not refused", R, x, 0);
  }
  for (int pattern = 0; pattern < PATTERNS; ++pattern) {
    double se[2][2] = {{0, 0}, {0, 0}};  // [normal / Gauss][FP64 / fixed] sums of squared errors
    for (int i = 0; i < 20000; ++i) {
      const int shift = (int)(rng() % 400) - 200;
      draw(pattern, R, buf);
      // errors in units of the sum of the terms' magnitudes, which bounds a chain's
      long double x[2] = {0.0L, 0.0L}, top[2] = {0.0L, 0.0L};
      for (int t = 0; t < R; ++t)
        for (int q = 0; q < 2; ++q) {
          const long double term = X.F[q ? 2 * K - t : t] * buf[t];
          x[q] += term;
          top[q] += std::fabs(term);
        }
      if (!asedf::fix_normal<R, 2>(v, 1, out)) fail("refused", R, buf[0], pattern);
      for (int q = 0; q < 2; ++q) {
        const double d = (double)((lin(R, v, q == 1, X) - x[q]) / top[q]), f = (double)((out[q] - x[q]) / top[q]);
        se[0][0] += d * d;
        se[0][1] += f * f;
      }
      gauss(R, G, v, X, g2);
      if (!asedf::fix_gauss<R, G>(v, 1, g1)) fail("refused at the Gauss points", R, buf[0], pattern);
      for (int g = 0; g < (G + 1) / 2; ++g) {
        long double E = X.E[g][0] * v[0], O = 0.0L;
        for (int t = 1; t <= K; ++t) {
          E += X.E[g][t] * ((long double)v[t] + v[-t]);
          O += X.O[g][t] * ((long double)v[t] - v[-t]);
        }
        for (int m = 0; m < (2 * g + 1 == G ? 1 : 2); ++m) {
          const int q = m ? G - 1 - g : g;
          const long double e = 2 * g + 1 == G ? E : m ? E - O : E + O;
          long double all = std::fabs(X.E[g][0] * v[0]);
          for (int t = 1; t <= K; ++t) {
            const long double a = X.E[g][t], b = m ? -X.O[g][t] : X.O[g][t];
            all += std::fabs((a + b) * v[t]) + std::fabs((a - b) * v[-t]);
          }
          const double d = (double)((g2[q] - e) / all), f = (double)((g1[q] - e) / all);
          se[1][0] += d * d;
          se[1][1] += f * f;
        }
      }
      // mirrored data swap the points, negated data negate them, a power of two scales them: to the bit
      for (int t = 0; t < R; ++t) { rev[t] = buf[R - 1 - t]; neg[t] = std::ldexp(-buf[t], shift); }
      asedf::fix_normal<R, 2>(rev + K, 1, o2);
      if (!same(out[0], o2[1]) || !same(out[1], o2[0])) fail("mirrored", R, out[0], o2[1]);
      asedf::fix_normal<R, 1>(v, -1, o2);
      if (!same(out[1], o2[0])) fail("one point", R, out[1], o2[0]);
      asedf::fix_normal<R, 2>(neg + K, 1, o2);
      if (out[0] != std::ldexp(-o2[0], -shift) || out[1] != std::ldexp(-o2[1], -shift)) fail("negated", R, out[0], o2[0]);
      asedf::fix_gauss<R, G>(neg + K, 1, g2);
      for (int q = 0; q < G; ++q)
        if (g1[q] != std::ldexp(-g2[q], -shift)) fail("negated Gauss point", R, g1[q], g2[q]);
    }
    std::printf("order %d, %s: rms error / FP64's: normal %.3f Gauss %.3f\n", R, kName[pattern],
                std::sqrt(se[0][1] / se[0][0]), std::sqrt(se[1][1] / se[1][0]));
    if (!(se[0][1] <= se[0][0]) || !(se[1][1] <= se[1][0])) fail("error above FP64's", R, pattern, 0);
  }
}

int main() {
  check<3>(kExact[0]);
  check<5>(kExact[1]);
  check<7>(kExact[2]);
  check<9>(kExact[3]);
  if (bad) std::printf("bad %ld\n", bad);
  else std::printf("ok\n");
  return bad != 0;
}
