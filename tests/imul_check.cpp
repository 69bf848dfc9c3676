// The integer-unit products of ase_df_imul.cuh compiled for the host, against the host's FP64
// product bit for bit: random significands, short ones (exact products and ties), all-ones ones,
// exponents to the ends of the range each function is stated for, zeros where they may be.
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <random>

#define __device__
#define __forceinline__ inline
static inline long long bits_of(double x) { long long b; std::memcpy(&b, &x, 8); return b; }
static inline long long __double_as_longlong(double x) { return bits_of(x); }
static inline int __double2hiint(double x) { return (int)(bits_of(x) >> 32); }
static inline int __double2loint(double x) { return (int)bits_of(x); }
static inline double __hiloint2double(int h, int l) {
  const unsigned long long b = ((unsigned long long)(unsigned)h << 32) | (unsigned)l;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}
static inline unsigned __funnelshift_l(unsigned lo, unsigned hi, unsigned s) {
  return (s & 31u) ? (hi << (s & 31u)) | (lo >> (32u - (s & 31u))) : hi;
}
#include "ase_df_imul.cuh"

static std::mt19937_64 rng(20241008);

// a normal double of binary exponent -lim .. lim
static double draw(int lim) {
  const uint64_t k = rng();
  uint64_t m = rng() & 0xfffffffffffffull;
  if ((k & 3u) == 0) { const int z = (int)((k >> 2) % 53); m = m >> z << z; }
  if ((k >> 8 & 7u) == 0) m |= 0xffffffffff000ull;
  if ((k >> 11 & 15u) == 0) m = 0;
  const uint64_t e = 1023 + (uint64_t)((int64_t)((k >> 16) % (2 * lim + 1)) - lim);
  const uint64_t b = (k & (1ull << 63)) | e << 52 | m;
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}

static long bad = 0;
static void same(const char* what, double x, double y, double got, double want) {
  if (bits_of(got) != bits_of(want) && bad++ < 5) std::printf("%s: %a * %a = %a, not %a\n", what, x, y, got, want);
}

int main() {
  long n = 0, ties = 0;
  for (int i = 0; i < 4000000; ++i, ++n) {
    const double x = draw(510), y = draw(510);
    same("imul", x, y, asedf::imul(x, y), x * y);
    same("imul_z", x, y, asedf::imul_z(x, y), x * y);
    const __int128 p = (__int128)((bits_of(x) & 0xfffffffffffffll) | 1ll << 52) * ((bits_of(y) & 0xfffffffffffffll) | 1ll << 52);
    const int sh = (p >> 105) ? 53 : 52;
    ties += (p & (((__int128)1 << sh) - 1)) == ((__int128)1 << (sh - 1));
  }
  for (const double z : {0.0, -0.0})
    for (int i = 0; i < 1000; ++i, ++n) {
      const double y = draw(300);
      same("imul_z of zero", z, y, asedf::imul_z(z, y), z * y);
    }
  // the ranges
  for (const double x : {0.0, -0.0}) bad += !asedf::imul_any(x) || asedf::imul_pos(x);
  for (const double x : {0x1p-64, 1.0, 0x1.fffffffffffffp64}) bad += !asedf::imul_pos(x) || asedf::imul_pos(-x);
  for (const double x : {0x1.fffffffffffffp-65, 0x1p65, 1.0 / 0.0, 0.0 / 0.0, 0x1p-1074}) bad += asedf::imul_pos(x);
  for (const double x : {0x1p-128, -0x1.fffffffffffffp128, -3.0}) bad += !asedf::imul_any(x);
  for (const double x : {0x1p-129, 0x1p129, -1.0 / 0.0, 0.0 / 0.0, 0x1p-1074, -0x1p-1030}) bad += asedf::imul_any(x);
  if (bad || ties < 1000) {
    std::printf("bad %ld, ties %ld\n", bad, ties);
    return 1;
  }
  std::printf("ok %ld ties %ld\n", n, ties);
  return 0;
}
