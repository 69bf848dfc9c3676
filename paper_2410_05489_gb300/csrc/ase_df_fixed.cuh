// Linear reconstructions in fixed point on the integer units.
//
// Why: this part issues FP64 at 1.6 lanes per cycle per SM (20 cycles a warp instruction,
// whatever the operation) and 32 x 32 -> 64 bit multiply-adds at 54, beside each other.  The
// linear branches of Algorithm 1 are contractions of 3 to 9 cell averages with constant
// weights, so they can leave the FP64 pipe to the Gauss-point flux: the 1024^2 order-9 sweep
// spent 321 of its 586 FP64 instructions per face on them.
//
// The values of a component in a tile share one exponent e (the largest of theirs):
//   v = M 2^(e - 1023 - 56), |M| < 2^57,
// so M keeps 4 bits below the last bit of a double of exponent e.  Weights are integers in
// units of 2^-56 that sum to 2^56 exactly (constant data are reproduced), split like M into
// limbs of 28 bits, w = wh 2^28 + wl with |wl| <= 2^27.  With M = mh 2^28 + ml,
//   sum w M / 2^56 = sum mh wh + (sum mh wl + ml wh) / 2^28 + (sum ml wl) / 2^56,
// and the last sum, below half a unit of M per term, is left out: three multiply-adds per
// term into two 64-bit sums, with an error of about a unit, 2^-56 of the tile's largest value
// (a chain of nine FP64 multiply-adds makes up to 2^-51 of it).
// Bounds: |value| <= 1.79 |M| for one reconstruction (the weights' absolute sum at order 9), so a
// normal reconstruction stays below 2^57.9, its tangential sums S = W_t + W_-t below 2^58.9
// (their high limb below 2^31), and the two 64-bit sums below 2^62.
#pragma once

#include "ase_df_device.cuh"

namespace asedf {
namespace {

constexpr int kFixBits = 56;  // fraction bits of M at the shared exponent, and of the weights
constexpr int kLimb = 28;
// Tiles with a larger biased exponent (values above 2^240) take the FP64 path, whose nonlinear
// weights overflow there.
constexpr int kFixMaxExp = 1023 + 240;
// The shared exponents serve a tile whose density and energy stay within this many binades: the
// smallest value then still has 52 bits above the unit of M.
constexpr int kFixRange = 4;

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

__device__ __forceinline__ Limbs fix_split(long long m) {
  return Limbs{(int)(m >> kLimb), (int)m & ((1 << kLimb) - 1)};
}

// Two-limb sum of products; the rounding half of the final shift is the starting value.
struct FixSum {
  long long hh, mid;
};
__device__ __forceinline__ FixSum fix_zero() { return FixSum{0ll, 1ll << (kLimb - 1)}; }
__device__ __forceinline__ void fix_mad(FixSum& s, Limbs m, int wh, int wl) {
  s.hh += (long long)m.h * wh;
  s.mid += (long long)m.h * wl;
  s.mid += (long long)m.l * wh;
}
__device__ __forceinline__ long long fix_value(FixSum s) { return s.hh + (s.mid >> kLimb); }

// Biased exponent of |x| from its high word (sign cleared).
__device__ __forceinline__ int exp_of(int abs_hi) { return (int)((unsigned)abs_hi >> 20); }

// The exponent values of largest biased exponent emax are kept at: not below 64, so that zeros
// and subnormals (far more than 57 binades below) become 0.
__device__ __forceinline__ int fix_exponent(int emax) { return emax < 64 ? 64 : emax; }

// M of a finite double at shared exponent e (biased exponent of x at most e + 1): the 53-bit
// significand shifted into place, truncated toward zero, sign applied to both limbs.
__device__ __forceinline__ Limbs fix_from_double(double x, int e) {
  const long long b = dbits(x);
  const int hi = (int)(b >> 32);
  int d = e + 1 - ((hi >> 20) & 0x7ff);
  d = d > 63 ? 63 : d;
  const unsigned long long sig =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)b) << (kFixBits - 51);
  const unsigned long long m = sig >> d;
  const int s = hi >> 31;
  const int h = (int)(m >> kLimb), l = (int)m & ((1 << kLimb) - 1);
  return Limbs{(h ^ s) - s, (l ^ s) - s};
}

__device__ __forceinline__ long long fix_join(Limbs m) { return ((long long)m.h << kLimb) + m.l; }

// The double nearest to R 2^(e - 1023 - 56), |R| < 2^62, 64 <= e <= 2046 - 62 (ties away from zero).
__device__ __forceinline__ double fix_to_double(long long R, int e) {
  const long long s = R >> 63;
  const unsigned long long a = (unsigned long long)((R ^ s) - s);
  // leading bit from a truncating conversion of the upper (or only) non-zero word
  const unsigned ah = (unsigned)(a >> 32);
  const unsigned w = ah != 0u ? ah : (unsigned)a;
  const int lead = (__float_as_int(__uint2float_rz(w)) >> 23) - (ah != 0u ? 95 : 127);  // for a != 0
  const unsigned long long m = ((a << ((62 - lead) & 63)) + 0x200u) >> 10;  // 53 bits, or 2^53
  const unsigned hi = (unsigned)(m >> 32) + ((unsigned)(e + lead - kFixBits - 1) << 20);
  const unsigned long long bits = (unsigned long long)(hi | ((unsigned)s & 0x80000000u)) << 32 | (unsigned)m;
  return __longlong_as_double(a == 0ull ? 0ll : (long long)bits);
}

}  // namespace
}  // namespace asedf
