// Products of doubles formed on the integer units, to the bit.
//
// Why: FP64 issues at 2 lanes per cycle per SM at most here.  A correctly rounded product takes four
// 32 x 32 -> 64 bit multiply-adds and some 24 other integer instructions, about 0.4 cycles a lane
// beside an FP64 pipe that works on (0.5 to 0.6 a lane).  So products that are no part of a fused multiply-add leave the FP64 pipe where
// it is the bound; where latency is (few warps on an SM), the FP64 instruction stays the shorter.
#pragma once

#include <cuda_runtime.h>

namespace asedf {
namespace {

__device__ __forceinline__ unsigned hi_word(double x) { return (unsigned)__double2hiint(x); }
__device__ __forceinline__ unsigned lo_word(double x) { return (unsigned)__double2loint(x); }

// x * y rounded to nearest, ties to even, for normal x, y with a normal product: the same bits as
// the FP64 unit's.  The significands, 53 bits of x and 53 of y shifted up by 11, multiply in four
// 32 x 32 -> 64 bit products to T 2^64 + f, T of 52 or 53 bits; T is shifted to 53 bits and
// rounded on f.  Signs and exponents are added in place: the carry of the exponents' sum into the
// sign bit leaves again with the bias.
__device__ __forceinline__ double imul(double x, double y) {
  const unsigned xh = hi_word(x), xl = lo_word(x), yh = hi_word(y), yl = lo_word(y);
  const unsigned a1 = (xh & 0xfffffu) | 0x100000u;
  const unsigned b1 = __funnelshift_l(yl, yh, 11) | 0x80000000u, b0 = yl << 11;
  const unsigned long long p00 = (unsigned long long)xl * b0;
  const unsigned long long p01 = (unsigned long long)xl * b1 + (p00 >> 32);
  const unsigned long long p10 = (unsigned long long)a1 * b0 + (unsigned)p01;
  const unsigned long long t = (unsigned long long)a1 * b1 + (p01 >> 32) + (p10 >> 32);
  const unsigned th = (unsigned)(t >> 32), tl = (unsigned)t, f1 = (unsigned)p10, f0 = (unsigned)p00;
  const unsigned s = (th >> 20) ^ 1u;  // 1: 52 bits
  const unsigned rh = __funnelshift_l(tl, th, s), rl = __funnelshift_l(f1, tl, s), f = __funnelshift_l(f0, f1, s);
  const unsigned long long r = (((unsigned long long)rh << 32) | rl) + (f >> 31);
  unsigned lo = (unsigned)r;
  if (f == 0x80000000u && f0 == 0u) lo &= ~1u;
  const unsigned hi = (unsigned)(r >> 32) + ((xh & 0xfff00000u) + (yh & 0xfff00000u) - (1023u << 20)) - (s << 20);
  return __hiloint2double((int)hi, (int)lo);
}

__device__ __forceinline__ unsigned long long dbits_abs(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7fffffffffffffffull;
}

// The same where x may be zero.
__device__ __forceinline__ double imul_z(double x, double y) {
  const double r = imul(x, y);
  return (hi_word(x) & 0x7fffffffu) != 0u ? r : __hiloint2double((int)((hi_word(x) ^ hi_word(y)) & 0x80000000u), 0);
}

// Operands for which the products of a Gauss point stay normal: positive within 2^-64 .. 2^64,
// and zero or within 2^-128 .. 2^128 in magnitude.
__device__ __forceinline__ bool imul_pos(double x) { return (hi_word(x) >> 20) - (1023u - 64u) <= 128u; }
__device__ __forceinline__ bool imul_any(double x) {
  return ((hi_word(x) >> 20) & 0x7ffu) - (1023u - 128u) <= 256u || (dbits_abs(x) == 0ull);
}

// A product of a Gauss point; lf_mulz: x may be zero.
template <bool INT>
__device__ __forceinline__ double lf_mul(double x, double y) {
  return INT ? imul(x, y) : x * y;
}
template <bool INT>
__device__ __forceinline__ double lf_mulz(double x, double y) {
  return INT ? imul_z(x, y) : x * y;
}

}  // namespace
}  // namespace asedf
