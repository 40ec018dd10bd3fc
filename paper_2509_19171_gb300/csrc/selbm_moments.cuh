// Node moments in 64-bit fixed point.
//
// rho - rho0 and rho u of a node are sums of its populations with velocity components 0, +-1.
// In FP64 they are about 65 additions a node on a pipe that issues two a clock and SM; the
// populations' common-scale integers add exactly on the integer pipe, and only the four sums
// return to FP64 (FP32 states are summed the same way: their sums are FP64 too).
#pragma once
#include "selbm_collide.cuh"
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

// ---------------------------------------------------------------------------
// BGK collision of one node in fixed point (FP64 form)
// ---------------------------------------------------------------------------
// With j = rho u and v = u + 2 kappa a (a the acceleration, kappa = (1/omega - 1/2) dt), the
// collision of Sec. 2.1 with F** is
//   f* = f + omega (t X - f),  X = drho + 3 e.j + 4.5 e e : P - 1.5 tr P,  P = (j v + v j) / 2,
// since rho (e.u)^2 = e e : (j u), and F** = t (9 (e.u)(e.F) - 3 u.F) with F = rho a enters f* as
// (1/omega - 1/2) dt omega F**.  The populations become integers at the node's largest exponent
// (rounded to nearest), moments and X are exact integer sums, and each population takes two
// fixed-point products (t and omega): about 60 integer instructions where the FP64 form takes 12
// FP64 ones, at 32 times their issue cost.  rho, 1 / rho and u stay FP64.
// Nodes beyond the integers' range (|v| >= 1/4, a density or momentum far above the largest
// deviation, infinities, NaN) take the FP64 collision.
struct CollideFix {
  Limb t[4];        // t_c / 2 times 2^64 by speed class
  Limb w;           // omega times 2^61
  double kappa2;    // 2 kappa
};
inline CollideFix make_collide_fix(const double *t_class, double omega, double dt) {
  CollideFix c{};
  for (int k = 0; k < 4; ++k) c.t[k] = limbs((long long)std::llrint(std::ldexp(0.5 * t_class[k], 64)));
  c.w = limbs((long long)std::llrint(std::ldexp(omega, 61)));
  c.kappa2 = 2.0 * (1.0 / omega - 0.5) * dt;
  return c;
}
template <int LAT>
CollideFix make_collide_fix(double omega, double dt) {
  constexpr VelTab V = LT<LAT>::v;
  double t[4] = {0, 0, 0, 0};
  for (int a = 0; a < V.Q; ++a) t[V.e[a][0] * V.e[a][0] + V.e[a][1] * V.e[a][1] + V.e[a][2] * V.e[a][2]] = V.t[a];
  return make_collide_fix(t, omega, dt);
}

// what the relaxation of a node's populations needs
struct NodeRelax {
  long long base, P[3], S[3], j[3];
  int em;           // exponent of the node's integers; 0: beyond their range (FP64 collision)
};

// integers, moments and products of one node (q: the populations at the node's scale); returns rho
template <int LAT, typename Load>
__device__ __forceinline__ double collide_moments(const CollideFix &cf, double rho0, const double (&acc)[3], bool forced,
                                                  Load load, long long (&q)[LT<LAT>::v.Q], NodeRelax &r) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, DIM = V.D, SH = 1;              // |q| <= 2^54
  int em = kMinExp;
  {
    double g[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) { g[a] = load(a); em = max(em, exp_of(g[a])); }
#pragma unroll
    for (int a = 0; a < Q; ++a) q[a] = to_fixed_rn<SH>(g[a], em);
  }
  long long sr = 0, sj[3] = {0, 0, 0};
  static_for<0, Q>([&](auto ac) {
    constexpr int a = decltype(ac)::value, o = LT<LAT>::v.opp[a];
    if constexpr (o == a) {
      sr += q[a];
    } else if constexpr (o > a) {
      const long long d = q[a] - q[o];
      sr += q[a] + q[o];
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (V.e[a][k] > 0) sj[k] += d;
        else if (V.e[a][k] < 0) sj[k] -= d;
      }
    }
  });
  const int ex = em - (1023 + 52 + SH);
  const double rho = rho0 + from_fixed(sr, ex);
  const double inv = 1.0 / rho;
  double v[3] = {0, 0, 0};
  int ev = 0;
  long long js = 0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    v[k] = from_fixed(sj[k], ex) * inv;
    if (forced) v[k] += cf.kappa2 * acc[k];
    ev = max(ev, exp_of(v[k]));
    js += sj[k] < 0 ? -sj[k] : sj[k];
  }
  const long long sra = sr < 0 ? -sr : sr;
  r.em = em == 2047 || ev > 1020 || sra >= (1ll << 60) || js >= (3ll << 57) ? 0 : em;
  // P_kk and S_kl = 2 P_kl
  Limb lj[3], lv[3];
#pragma unroll
  for (int k = 0; k < DIM; ++k) { lj[k] = limbs(sj[k]); lv[k] = limbs(to_fixed<6>(v[k], 1022)); }   // v 2^59
  long long tr = 0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    Fix128 s{0, 0};
    fix_mac(s, lj[k], lv[k]);
    r.P[k] = fix_top<5>(s);
    r.j[k] = sj[k];
    tr += r.P[k];
  }
#pragma unroll
  for (int k = 0; k < DIM; ++k)
#pragma unroll
    for (int l = k + 1; l < DIM; ++l) {
      Fix128 s{0, 0};
      fix_mac(s, lj[k], lv[l]);
      fix_mac(s, lj[l], lv[k]);
      r.S[k + l - 1] = fix_top<5>(s);                    // xy, xz, yz
    }
  r.base = 2 * sr - 3 * tr;
  return rho;
}

// relaxed populations a and its opposite (a <= opposite) of a node within the integers' range
template <int LAT, int a, typename Store>
__device__ __forceinline__ void collide_pair(const CollideFix &cf, const NodeRelax &r, long long qa, long long qo, Store store) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int DIM = V.D, o = LT<LAT>::v.opp[a], ea = V.e[a][0], eb = V.e[a][1], ec = V.e[a][2];
  constexpr int cls = ea * ea + eb * eb + ec * ec;
  long long even = 0, ej = 0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    if (V.e[a][k] != 0) even += r.P[k];
    if (V.e[a][k] > 0) ej += r.j[k];
    else if (V.e[a][k] < 0) ej -= r.j[k];
#pragma unroll
    for (int l = k + 1; l < DIM; ++l) {
      if (V.e[a][k] * V.e[a][l] > 0) even += r.S[k + l - 1];
      else if (V.e[a][k] * V.e[a][l] < 0) even -= r.S[k + l - 1];
    }
  }
  const long long e9 = r.base + 9 * even, o6 = 6 * ej;
  auto relax = [&](int b, long long q, long long x2) {
    Fix128 f{0, 1ll << 31};                              // + 1/2: rounded to nearest
    fix_mac(f, cf.t[cls], limbs(x2));
    Fix128 w{0, 1ll << 28};
    fix_mac(w, cf.w, limbs(fix_top<0>(f) - q));
    store(b, from_fixed(q + fix_top<3>(w), r.em - (1023 + 52 + 1)));
  };
  relax(a, qa, e9 + o6);
  if constexpr (o != a) relax(o, qo, e9 - o6);
}

// load(a) / store(a, value) of the node's deviations (load before any store); returns rho
template <int LAT, typename Load, typename Store>
__device__ __forceinline__ double collide_fixed(const CollideFix &cf, double rho0, double omega, double dt, double half_dt,
                                                const double (&acc)[3], bool forced, Load load, Store store) {
  constexpr int Q = LT<LAT>::v.Q;
  long long q[Q];
  NodeRelax r;
  const double rho = collide_moments<LAT>(cf, rho0, acc, forced, load, q, r);
  if (r.em == 0) {
    double g[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) g[a] = load(a);
    const double rs = bgk_collide<double, LAT>(g, rho0, omega, dt, half_dt, acc, forced);
#pragma unroll
    for (int a = 0; a < Q; ++a) store(a, g[a]);
    return rs;
  }
  static_for<0, Q>([&](auto ac) {
    constexpr int a = decltype(ac)::value, o = LT<LAT>::v.opp[a];
    if constexpr (o >= a) collide_pair<LAT, a>(cf, r, q[a], q[o], store);
  });
  return rho;
}

}  // namespace slb
