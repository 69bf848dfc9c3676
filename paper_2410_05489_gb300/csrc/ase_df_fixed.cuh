// Linear reconstructions in fixed point on the integer units.
//
// Why: this part issues FP64 at 2 lanes per cycle per SM at most and 32 x 32 -> 64 bit
// multiply-adds at 54, beside each other.  The
// linear branches of Algorithm 1 are contractions of 3 to 9 cell averages with constant
// weights, so they can leave the FP64 pipe to the Gauss-point flux: of the 475 FP64 instructions
// of an order-9 face in a smooth flow, whose products of the Gauss points run on the integer units, they are 321.
//
// The values of ONE stencil share one exponent e, that of the largest:
//   |v| = M 2^(e - 1023 - 56), M < 2^57.
// A stencil whose values have one sign and lie within kFixRange binades is exact in M, so the result
// is a function of the stencil's values alone, whichever tile or launch evaluates it, and an error
// is relative to these values.  (A momentum that changes sign in the stencil, or a value far below its
// neighbours, takes the FP64 chain; zeros throughout give zero.)
// Weights are integers in units of 2^-56 that sum to 2^56 exactly.  The sum is therefore formed as
//   M_0 + sum w_t (M_t - M_0) / 2^56
// which reproduces constant data to the bit.  With differences and weights in limbs of 28 bits,
// d = dh 2^28 + dl and w = wh 2^28 + wl, |wl| <= 2^27,
//   sum w d / 2^56 = sum dh wh + (sum dh wl + dl wh) / 2^28 + (sum dl wl) / 2^56,
// and the last sum, below half a unit of M per term, is left out: three multiply-adds per
// term into two 64-bit sums and one rounding to double.  Measured against exact sums over stencils that span
// 0 to kFixRange binades (host test), the rms error is 0.4 to 0.7 of the FP64 chain's.
// Bounds: |M_t - M_0| < 2^57, so its high limb is below 2^29, that of (M_t - M_0) + (M_-t - M_0) below
// 2^30; the weights' absolute sum without the centre's is below 1.1, so results stay below 2^59
// and both 64-bit sums below 2^61.
#pragma once

#include <cuda_runtime.h>

namespace asedf {
namespace {

constexpr int kFixBits = 56;  // fraction bits of M at the stencil's exponent, and of the weights
constexpr int kLimb = 28;
// Biased exponents of a stencil's largest value: not below 64 (results stay normal) nor beyond 2^240
// (infinities and NaN, and values whose nonlinear weights overflow elsewhere).
constexpr int kFixMinExp = 64, kFixMaxExp = 1023 + 240;
// Largest difference between the exponents of a stencil.
constexpr int kFixRange = 3;

// Weights of the order-r linear branch (index (r - 3) / 2), high and low limbs:
//   f: W_t, t = -k..k, at xi = 0 (xi = -1 is its mirror image);
//   e, o: even and odd parts at the Gauss-point pair g (E = e_0 W_0 + sum e_t (W_t + W_-t),
//   O = sum o_t (W_t - W_-t), values E +- O), as Tables::se, so.
struct FixWeights {
  int fh[9], fl[9];
  int eh[2][5], el[2][5];
  int oh[2][5], ol[2][5];
};

__constant__ FixWeights kFixW[4] = {
    {{-44739243, 223696213, 89478485, 0, 0, 0, 0, 0, 0},
     {89478485, 89478486, 89478485, 0, 0, 0, 0, 0, 0},
     {{290805077, -11184811, 0, 0, 0}, {0, 0, 0, 0, 0}},
     {{89478486, 89478485, 0, 0, 0}, {0, 0, 0, 0, 0}},
     {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}},
     {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}}},  // order 3
    {{8947849, -58161015, 210274441, 120795955, -13421773, 0, 0, 0, 0},
     {-125269879, -125269879, -125269880, 53687091, 53687091, 0, 0, 0, 0},
     {{268062629, 248551, -62138, 0, 0}, {0, 0, 0, 0, 0}},
     {{-5965232, 93455307, 43745037, 0, 0}, {0, 0, 0, 0, 0}},
     {{0, -53812945, 7533812, 0, 0}, {0, 0, 0, 0, 0}},
     {{0, -110136825, 95949792, 0, 0}, {0, 0, 0, 0, 0}}},  // order 5
    {{-1917396, 15978301, -64552336, 203883120, 136774256, -24287017, 2556528, 0, 0},
     {-30678338, -12782641, 40904450, 40904452, 40904450, -120156823, 40904450, 0, 0},
     {{241508823, 15217734, -1903974, 149557, 0}, {302099739, -19026661, 2381765, -187246, 0}},
     {{63095114, -46426551, -91666873, -27671861, 0}, {-48574036, -48574035, 130382936, 76695845, 0}},
     {{0, -80883019, 17402520, -1968108, 0}, {0, 0, 0, 0, 0}},
     {{0, 57617975, -73794642, 71957663, 0}, {0, 0, 0, 0, 0}}},  // order 7
    {{426088, -4367402, 21197879, -68280606, 200154850, 146467759, -32489212, 5858710, -532610},
     {6817408, -69878436, 70730612, -18747873, -18747873, -72434964, 17043521, 93739366, -8521761},
     {{225411367, 24812032, -3767748, 503933, -36173}, {291384530, -13234749, 2009714, -268796, 19294}},
     {{-93549424, 102065331, 118498354, -93484201, 53912956}, {-19691606, 86082520, -95217202, -81399035, 100379520}},
     {{0, -95118404, 24980278, -4815359, 453512}, {0, -40158090, 11704927, -2316352, 220388}},
     {{0, -99098226, -24657156, -60676763, -93229744}, {0, 25320571, -52510059, -32973009, -63827788}}},  // order 9
};

struct Limbs {
  int h, l;
};

// M of the magnitude of a normal double; k = 8 - (e - its exponent), 4 < k <= 8.
__device__ __forceinline__ Limbs fix_from_double(int hi, int lo, int k) {
  const unsigned a = (unsigned)((hi & 0xfffff) | 0x100000);
  return Limbs{(int)__funnelshift_l((unsigned)lo, a, k), (int)(((unsigned)lo << k) >> 4)};
}

// Two-limb sum, in units of 1 and 2^-28.
struct FixSum {
  long long hh, mid;
};
__device__ __forceinline__ void fix_mad(FixSum& s, Limbs d, int wh, int wl) {
  s.hh += (long long)d.h * wh;
  s.mid += (long long)d.h * wl;
  s.mid += (long long)d.l * wh;
}

// The double nearest to +- s 2^(e - 1023 - 56), |s| < 2^61, kFixMinExp <= e <= kFixMaxExp; sign: 0, or
// the sign bit of the stencil's values.
__device__ __forceinline__ double fix_to_double(FixSum s, int e, unsigned sign) {
  const long long R = s.hh + ((s.mid + (1ll << (kLimb - 1))) >> kLimb), n = R >> 63;
  const unsigned long long a = (unsigned long long)((R ^ n) - n);
  // leading bit from a truncating conversion of the upper (or only) non-zero word
  const unsigned ah = (unsigned)(a >> 32);
  const unsigned w = ah != 0u ? ah : (unsigned)a;
  const int lead = (__float_as_int(__uint2float_rz(w)) >> 23) - (ah != 0u ? 95 : 127);  // for a != 0
  const unsigned long long m = ((a << ((62 - lead) & 63)) + 0x200u) >> 10;  // 53 bits, or 2^53
  const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(e + lead - kFixBits - 1) << 20);
  const unsigned long long bits = (unsigned long long)(hi | (((unsigned)n & 0x80000000u) ^ sign)) << 32 | (unsigned)m;
  return __longlong_as_double(a == 0ull ? 0ll : (long long)bits);
}

// A stencil of 2 K + 1 values in fixed point.
template <int K>
struct FixStencil {
  int e;
  unsigned sign;     // sign bit of the values
  long long m0;      // the centre
  Limbs p[K], m[K];  // W_t - W_0 and W_-t - W_0, t = 1 .. K

  // v points at W_0, W_t at v[t vs].  Returns 1; 0 when the stencil does not fit; -1 when it is all zeros.
  __device__ __forceinline__ int load(const double* v, int vs) {
    int hi[2 * K + 1], lo[2 * K + 1];
    int mx = -0x7fffffff, mn = 0x7fffffff;  // of the exponents, less 2048 for negative values
#pragma unroll
    for (int t = 0; t <= 2 * K; ++t) {
      const long long b = __double_as_longlong(v[(t - K) * vs]);
      hi[t] = (int)(b >> 32);
      lo[t] = (int)b;
      mx = max(mx, hi[t] >> 20);
      mn = min(mn, hi[t] >> 20);
    }
    e = mx & 0x7ff;
    sign = (unsigned)mx & 0x80000000u;
    if (mx - mn > kFixRange || (unsigned)(e - kFixMinExp) > (unsigned)(kFixMaxExp - kFixMinExp)) {
      int any = 0;
#pragma unroll
      for (int t = 0; t <= 2 * K; ++t) any |= (hi[t] & 0x7fffffff) | lo[t];
      return any == 0 ? -1 : 0;
    }
    const Limbs c = fix_from_double(hi[K], lo[K], (hi[K] >> 20) - mx + 8);
    m0 = (long long)c.h * (1 << kLimb) + c.l;
#pragma unroll
    for (int t = 1; t <= K; ++t) {
      const Limbs a = fix_from_double(hi[K + t], lo[K + t], (hi[K + t] >> 20) - mx + 8);
      const Limbs b = fix_from_double(hi[K - t], lo[K - t], (hi[K - t] >> 20) - mx + 8);
      p[t - 1] = Limbs{a.h - c.h, a.l - c.l};
      m[t - 1] = Limbs{b.h - c.h, b.l - c.l};
    }
    return 1;
  }
};

// Order-R linear reconstruction at the upper face (xi = 0) of the stencil's cell and, with NP = 2,
// at the lower one (xi = -1: the mirrored weights).  Returns whether the stencil fits.
template <int R, int NP>
__device__ __forceinline__ bool fix_normal(const double* v, int vs, double* out) {
  constexpr int K = (R - 1) / 2;
  const FixWeights& F = kFixW[(R - 3) / 2];
  FixStencil<K> s;
  const int fit = s.load(v, vs);
  if (fit <= 0) {
#pragma unroll
    for (int q = 0; q < NP; ++q) out[q] = 0.0;
    return fit != 0;
  }
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    FixSum x{s.m0, 0ll};
#pragma unroll
    for (int t = 1; t <= K; ++t) {
      fix_mad(x, q == 0 ? s.p[t - 1] : s.m[t - 1], F.fh[K + t], F.fl[K + t]);
      fix_mad(x, q == 0 ? s.m[t - 1] : s.p[t - 1], F.fh[K - t], F.fl[K - t]);
    }
    out[q] = fix_to_double(x, s.e, s.sign);
  }
  return true;
}

// Gauss-point values of the order-R linear branch by the even and odd sums of lin_gauss_sym: the
// points eta and -1 - eta are E +- O.  Returns whether the stencil fits.
template <int R, int G>
__device__ __forceinline__ bool fix_gauss(const double* v, int vs, double* out) {
  constexpr int K = (R - 1) / 2;
  const FixWeights& F = kFixW[(R - 3) / 2];
  FixStencil<K> s;
  const int fit = s.load(v, vs);
  if (fit <= 0) {
#pragma unroll
    for (int q = 0; q < G; ++q) out[q] = 0.0;
    return fit != 0;
  }
#pragma unroll
  for (int g = 0; g < (G + 1) / 2; ++g) {
    FixSum E{s.m0, 0ll}, O{0ll, 0ll};
#pragma unroll
    for (int t = 1; t <= K; ++t)
      fix_mad(E, Limbs{s.p[t - 1].h + s.m[t - 1].h, s.p[t - 1].l + s.m[t - 1].l}, F.eh[g][t], F.el[g][t]);
    if (2 * g + 1 == G) {
      out[g] = fix_to_double(E, s.e, s.sign);  // middle point
    } else {
#pragma unroll
      for (int t = 1; t <= K; ++t)
        fix_mad(O, Limbs{s.p[t - 1].h - s.m[t - 1].h, s.p[t - 1].l - s.m[t - 1].l}, F.oh[g][t], F.ol[g][t]);
      out[g] = fix_to_double(FixSum{E.hh + O.hh, E.mid + O.mid}, s.e, s.sign);
      out[G - 1 - g] = fix_to_double(FixSum{E.hh - O.hh, E.mid - O.mid}, s.e, s.sign);
    }
  }
  return true;
}

}  // namespace
}  // namespace asedf
