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
// (1/omega - 1/2) dt omega F**.  The populations become integers at the node's largest exponent with
// kColShift bits below its last FP64 bit (rounded to nearest), moments are exact integer sums, X is
// formed in units of four (t <= 1/9 brings it back below one) and each population takes two
// fixed-point products (t and omega): about 60 integer instructions where the FP64 form takes 12
// FP64 ones, at 32 times their issue cost.  The change omega (t X - f) alone returns to FP64, times
// 2^w_shift so that a small omega keeps its bits, and is added to f: a population that is small next
// to the node's largest one keeps all of its own bits.  rho, 1 / rho and u stay FP64.  Taylor-Green 16^3,
// D3Q27: 244 us a launch (1.09 ms in FP64 arithmetic), ALU 58 % at 24 % warps.
// Nodes beyond the integers' range (|v| >= 1/4, a momentum far above the largest deviation,
// infinities, NaN) take the FP64 collision.
//
// Bounds, in units of the integers, m = 2^(53 + kColShift) above every |q|: |sum q| <= 27 m < 2^62;
// with js = |j_x| + |j_y| + |j_z| < 2^62 (2D: 2^61) and |v_k| < 1/4, |X| / 4 < 7.8 2^60, so that t X and
// omega (t X - q) stay below 2^63.
// The corner populations of D3Q27 (t = 1 / 216) are small next to a node's largest one and take three
// bits more.
constexpr int kColShift = 4;
constexpr int speed_class(const VelTab &v, int a) { return v.e[a][0] * v.e[a][0] + v.e[a][1] * v.e[a][1] + v.e[a][2] * v.e[a][2]; }
constexpr int fine_bits(int cls) { return cls == 3 ? 3 : 0; }
struct CollideFix {
  Limb t[4];        // t_c 2^66 by speed class (rest: 2^64)
  Limb w;           // omega times 2^(61 + w_shift), in [2^61, 2^62]
  int w_shift;
  double kappa2;    // 2 kappa
};
inline CollideFix make_collide_fix(const double *t_class, double omega, double dt) {
  CollideFix c{};
  for (int k = 0; k < 4; ++k) c.t[k] = limbs((long long)std::llrint(std::ldexp(t_class[k], k == 0 ? 64 : 66)));
  c.w_shift = std::max(0, std::min(60, -std::ilogb(omega)));
  c.w = limbs((long long)std::llrint(std::ldexp(omega, 61 + c.w_shift)));
  c.kappa2 = 2.0 * (1.0 / omega - 0.5) * dt;
  return c;
}
template <int LAT>
CollideFix make_collide_fix(double omega, double dt) {
  constexpr VelTab V = LT<LAT>::v;
  double t[4] = {0, 0, 0, 0};
  for (int a = 0; a < V.Q; ++a) t[speed_class(V, a)] = V.t[a];
  return make_collide_fix(t, omega, dt);
}

// a velocity below 1/4 as an integer times 2^62, and the largest momentum of the integers' range
__device__ __forceinline__ long long fix_velocity(double v) { return to_fixed_rn<9>(v, 1022); }
template <int DIM>
__device__ __forceinline__ bool fix_in_range(int em, int ev, long long js) {
  return em != 2047 && ev <= 1020 && js < (1ll << (DIM == 2 ? 61 : 62));
}
// j v in the integers' units, v from fix_velocity
__device__ __forceinline__ long long fix_product(const Fix128 &s) { return fix_top<2>(s); }
// X / 4 of the moving populations: sr / 4 + 3 ej / 4 + (9 even - 3 tr) / 8, each part rounded
__device__ __forceinline__ long long fix_quarter(long long x) { return (x + 2) >> 2; }
__device__ __forceinline__ long long fix_base4(long long sr, long long tr) { return fix_quarter(sr) - ((3 * tr + 4) >> 3); }
__device__ __forceinline__ long long fix_rest(long long sr, long long tr) { return sr - ((3 * tr + 1) >> 1); }
__device__ __forceinline__ long long fix_even4(long long even) { return even + ((even + 4) >> 3); }
// omega (t X - q) of one population, as FP64; t from CollideFix, x is X (rest) or X / 4, q has FINE bits
// more than x
template <int FINE = 0>
__device__ __forceinline__ double fix_change(const CollideFix &cf, const Limb &t, long long x, long long q, int em) {
  Fix128 f{0, 1ll << (31 - FINE)};                       // + 1/2: rounded to nearest
  fix_mac_full(f, t, limbs(x));
  Fix128 r{0, 1ll << 28};
  fix_mac_full(r, cf.w, limbs(fix_top<FINE>(f) - q));
  return from_fixed(fix_top<3>(r), em - (1023 + 52 + kColShift + FINE) - cf.w_shift);
}

// what the relaxation of a node's populations needs
struct NodeRelax {
  long long rest, base, P[3], S[3], j[3];
  int em;           // exponent of the node's integers; 0: beyond their range (FP64 collision)
};

// integers, moments and products of one node (q: the populations at the node's scale); returns rho
template <int LAT, typename Load>
__device__ __forceinline__ double collide_moments(const CollideFix &cf, double rho0, const double (&acc)[3], bool forced,
                                                  Load load, long long (&q)[LT<LAT>::v.Q], NodeRelax &r) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, DIM = V.D;
  int em = kMinExp;
  {
    double g[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) { g[a] = load(a); em = max(em, exp_of(g[a])); }
    static_for<0, Q>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      q[a] = to_fixed_rn<kColShift + fine_bits(speed_class(V, a))>(g[a], em);
    });
  }
  long long sr = 0, sj[3] = {0, 0, 0};
  static_for<0, Q>([&](auto ac) {
    constexpr int a = decltype(ac)::value, o = LT<LAT>::v.opp[a];
    if constexpr (o == a) {
      sr += q[a];
    } else if constexpr (o > a) {
      constexpr int fine = fine_bits(speed_class(V, a)), half = (1 << fine) >> 1;
      const long long d = (q[a] - q[o] + half) >> fine;
      sr += (q[a] + q[o] + half) >> fine;
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (V.e[a][k] > 0) sj[k] += d;
        else if (V.e[a][k] < 0) sj[k] -= d;
      }
    }
  });
  const int ex = em - (1023 + 52 + kColShift);
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
    js += (sj[k] < 0 ? -sj[k] : sj[k]) >> 2;             // quarters: three sums of 2^62 stay in range
  }
  r.em = fix_in_range<DIM>(em, ev, js * 4) ? em : 0;
  // P_kk and S_kl = 2 P_kl
  Limb lj[3], lv[3];
#pragma unroll
  for (int k = 0; k < DIM; ++k) { lj[k] = limbs(sj[k]); lv[k] = limbs(fix_velocity(v[k])); }
  long long tr = 0;
#pragma unroll
  for (int k = 0; k < DIM; ++k) {
    Fix128 s{0, 0};
    fix_mac(s, lj[k], lv[k]);
    r.P[k] = fix_product(s);
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
      r.S[k + l - 1] = fix_product(s);                   // xy, xz, yz
    }
  r.base = fix_base4(sr, tr);
  r.rest = fix_rest(sr, tr);
  return rho;
}

// relaxed populations a and its opposite (a <= opposite) of a node within the integers' range
template <int LAT, int a, typename Load, typename Store>
__device__ __forceinline__ void collide_pair(const CollideFix &cf, const NodeRelax &r, long long qa, long long qo,
                                             Load load, Store store) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int DIM = V.D, o = LT<LAT>::v.opp[a], cls = speed_class(V, a), fine = fine_bits(cls);
  if constexpr (o == a) {
    store(a, load(a) + fix_change(cf, cf.t[0], r.rest, qa, r.em));
  } else {
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
    const long long e4 = r.base + fix_even4(even), o4 = 3 * fix_quarter(ej);
    const double fa = load(a), fo = load(o);
    store(a, fa + fix_change<fine>(cf, cf.t[cls], e4 + o4, qa, r.em));
    store(o, fo + fix_change<fine>(cf, cf.t[cls], e4 - o4, qo, r.em));
  }
}

// load(a) / store(a, value) of the node's deviations (a population is loaded again before its store:
// from the cache, as its integer and its value do not both fit the registers); returns rho
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
    if constexpr (o >= a) collide_pair<LAT, a>(cf, r, q[a], q[o], load, store);
  });
  return rho;
}

}  // namespace slb
