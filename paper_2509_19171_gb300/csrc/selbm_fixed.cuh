// 64-bit fixed-point lines for the FP64 form.
//
// GB300 issues two FP64 operations per clock and SM (measured: DFMA 1.99 lanes/clk/SM, against
// 64 for 32-bit integer multiply-adds and 122 for FFMA), so an FP64 kernel is bound by the FP64
// pipe whatever else it does.  The line products of the scheme (derivative, filter) are dot
// products of one line's values with fixed coefficients: a block-scaled integer form is exact
// enough and runs on the integer pipes.  A value of a population tile becomes a signed 60-bit
// integer at the tile's largest exponent, a coefficient a signed integer of up to 62 bits, and a
// product is formed from 32-bit signed limbs,
//   C q / 2^64 = Ch Qh + (Ch Ql + Cl Qh) / 2^32 (+ Cl Ql / 2^64, below the last place kept),
// three IMAD.WIDE instead of one DFMA that costs 32 times an issue slot.  The dropped lowest products are
// at most a quarter of the sum's last place each, before the shift of a result by up to three bits: a line
// of n terms is off by at most n 2^-59 of (row sum of |coefficients|) x (tile's largest value), 2^-57 and
// less on average (figures in selbm_fixed_lines.cuh); where that matters the high word of the lowest
// product is added too.  The results return to FP64 rounded to nearest.
#pragma once
#include <cuda_runtime.h>

#include <cmath>
#include <algorithm>
#include <cstdint>

namespace slb {

// signed limbs of a 64-bit integer: q = hi 2^32 + lo, lo in [-2^31, 2^31)
struct Limb {
  int hi, lo;
};
__host__ __device__ __forceinline__ Limb limbs(long long q) {
  Limb l;
  l.lo = (int)(unsigned)(unsigned long long)q;
  l.hi = (int)(q >> 32) + (int)((unsigned)l.lo >> 31);
  return l;
}

// sums of Ch Qh and of the cross products; value = A 2^64 + B 2^32
struct Fix128 {
  long long A, B;
};
__device__ __forceinline__ void fix_mac(Fix128 &s, const Limb &c, const Limb &q) {
  s.A += (long long)c.hi * q.hi;
  s.B += (long long)c.hi * q.lo;
  s.B += (long long)c.lo * q.hi;
}
// adds C Q with the high word of the lowest product too: the sum is shifted up afterwards
__device__ __forceinline__ void fix_mac_full(Fix128 &s, const Limb &c, const Limb &q) {
  fix_mac(s, c, q);
  s.B += (long long)__mulhi(c.lo, q.lo);
}
// (A 2^64 + B 2^32) / 2^(64 - K), 0 <= K <= 31
template <int K>
__device__ __forceinline__ long long fix_top(const Fix128 &s) {
  return (long long)((unsigned long long)s.A << K) + (s.B >> (32 - K));
}

// bits of headroom: |q| < 2^(kFixBits) after to_fixed; two values add up without overflow
template <int n>
struct FixScale {
  // products of a line sum at most 2 ceil(n/2) cross terms of 2^31 2^(bits - 31): 63 bits
  static constexpr int SHIFT = n > 10 ? 5 : 6;          // mantissa (53 bits) shifted up by SHIFT
  static constexpr int BITS = 53 + SHIFT;                // |q| < 2^BITS
  // value = q 2^(emax - EXP0), emax the biased exponent of the tile's largest value
  static constexpr int EXP0 = 1023 + 52 + SHIFT;
};

// biased exponent of |v| (0 for zeros and subnormals, 2047 for infinities and NaN)
__device__ __forceinline__ int exp_of(double v) { return (__double2hiint(v) >> 20) & 0x7ff; }

// v at the tile's scale (emax >= exponent of v, emax >= kMinExp), truncated toward zero
constexpr int kMinExp = 64;    // smaller tiles (values below 2^-959) are taken at this scale
template <int SHIFT>
__device__ __forceinline__ long long to_fixed(double v, int emax) {
  const int hi = __double2hiint(v), lo = __double2loint(v);
  const int sh = min(emax - ((hi >> 20) & 0x7ff), 63);
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32 | (unsigned)lo) << SHIFT;
  const long long u = (long long)(m >> sh), s = (long long)(hi >> 31);
  return (u ^ s) - s;
}

// the same rounded to nearest (ties away from zero)
template <int SHIFT>
__device__ __forceinline__ long long to_fixed_rn(double v, int emax) {
  const long long q = to_fixed<SHIFT + 1>(v, emax), s = q >> 63;
  return (q - s) >> 1;                                   // |q| odd: away from zero
}

// the same beyond the range of normal FP64 numbers (out of line: the code of the usual case counts)
static __device__ __noinline__ double from_fixed_rare(long long r, int ex) { return scalbn((double)r, ex); }
// r 2^ex as FP64, rounded to nearest
__device__ __forceinline__ double from_fixed(long long r, int ex) {
  const long long s = r >> 63;
  unsigned long long a = (unsigned long long)((r ^ s) - s);
  const int lz = __clzll((long long)a);                  // 64 when r = 0
  a <<= (lz & 63);
  const unsigned long long mant = (a >> 11) + ((a >> 10) & 1ull);   // 2^52 .. 2^53
  const int E = 1086 - lz + ex;                          // biased exponent of the result
  if ((unsigned)(E - 1) >= 2045u) return r == 0 ? 0.0 : from_fixed_rare(r, ex);
  unsigned long long bits = ((unsigned long long)(unsigned)(E - 1) << 52) + mant;
  bits = r == 0 ? 0ull : bits;
  return __longlong_as_double((long long)(bits | ((unsigned long long)s & 0x8000000000000000ull)));
}

// g 2^k rounded to an integer, k chosen so that the largest |g| of the set stays below 2^bits
inline int fix_shift(double gmax, int bits) {
  if (!(gmax > 0.0)) return 0;
  int e;
  std::frexp(gmax, &e);                                  // gmax < 2^e
  return bits - e;
}
inline Limb fix_coef(double g, int k) { return limbs((long long)std::llrint(std::ldexp(g, k))); }

}  // namespace slb
