// Node moments in 64-bit fixed point.
//
// rho - rho0 and rho u of a node are sums of its populations with velocity components 0, +-1.
// In FP64 they are about 65 additions a node on a pipe that issues two a clock and SM; the
// populations' common-scale integers add exactly on the integer pipe, and only the four sums
// return to FP64 (FP32 states are summed the same way: their sums are FP64 too).
#pragma once
#include "selbm_fixed.cuh"
#include "selbm_lattice.cuh"

namespace slb {

constexpr int kSumShift = 5;   // |q| < 2^58: 27 of them stay below 2^63

__device__ __forceinline__ int moment_exp(double v) { return exp_of(v); }
__device__ __forceinline__ int moment_exp(float v) {
  const int e = (__float_as_int(v) >> 23) & 0xff;
  return e == 255 ? 2047 : (e == 0 ? 0 : e + 896);       // biased as an FP64 exponent
}
__device__ __forceinline__ long long moment_fixed(double v, int emax) { return to_fixed<kSumShift>(v, emax); }
__device__ __forceinline__ long long moment_fixed(float v, int emax) {
  // FP32 subnormals (below 2^-126) count as zero next to a node's other populations
  const int x = __float_as_int(v), e = (x >> 23) & 0xff;
  const int sh = e == 0 ? 63 : min(emax - e - 896, 63);
  const unsigned long long m = (unsigned long long)(unsigned)((x & 0x7fffff) | 0x800000) << (29 + kSumShift);
  const long long u = (long long)(m >> sh), s = (long long)(x >> 31);
  return (u ^ s) - s;
}

// FP64 value of a state entry without the FP64 pipe
__device__ __forceinline__ double wide(double v) { return v; }
__device__ __forceinline__ double wide(float v) {
  const unsigned x = __float_as_uint(v), e = (x >> 23) & 0xffu;
  if (e == 0u || e == 255u) return (double)v;
  return __hiloint2double((int)((x & 0x80000000u) | (((x & 0x7fffffffu) >> 3) + (896u << 20))), (int)(x << 29));
}

// drho = sum_a g_a, j = sum_a e_a g_a of one node's deviations; returns the number of
// non-finite populations (then the sums are FP64 sums)
template <int LAT, typename Real>
__device__ __forceinline__ int node_moments(const Real (&g)[LT<LAT>::v.Q], double &drho, double (&j)[3]) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, DIM = V.D;
  int em = kMinExp;
#pragma unroll
  for (int a = 0; a < Q; ++a) em = max(em, moment_exp(g[a]));
  j[0] = j[1] = j[2] = 0;
  if (em == 2047) {
    int bad = 0;
    drho = 0;
    static_for<0, Q>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      const double v = (double)g[a];
      bad += !isfinite(v);
      drho += v;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (V.e[a][k] > 0) j[k] += v;
        else if (V.e[a][k] < 0) j[k] -= v;
      }
    });
    return bad;
  }
  long long sr = 0, sj[3] = {0, 0, 0};
  static_for<0, Q>([&](auto ac) {
    constexpr int a = decltype(ac)::value, o = LT<LAT>::v.opp[a];
    if constexpr (o == a) {
      sr += moment_fixed(g[a], em);
    } else if constexpr (o > a) {
      const long long p = moment_fixed(g[a], em), m = moment_fixed(g[o], em), d = p - m;
      sr += p + m;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (V.e[a][k] > 0) sj[k] += d;
        else if (V.e[a][k] < 0) sj[k] -= d;
      }
    }
  });
  const int ex = em - (1023 + 52 + kSumShift);
  drho = from_fixed(sr, ex);
#pragma unroll
  for (int k = 0; k < DIM; ++k) j[k] = from_fixed(sj[k], ex);
  return 0;
}

}  // namespace slb
