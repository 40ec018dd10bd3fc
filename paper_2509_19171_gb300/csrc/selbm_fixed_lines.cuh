// Lines of the any-order kernels: sizes, coefficients, and the FP64 line operations in 64-bit fixed point
// (the FP32 ones are in selbm_lines.cuh).  `Host` holds D, w, Vm, Vinv and fixed_sigma (SplitHost).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "selbm_fixed.cuh"

namespace slb {

template <typename Real>
using LineVal = std::conditional_t<sizeof(Real) == 8, long long, float>;       // a line's value
template <typename Real>
using LineCoef = std::conditional_t<sizeof(Real) == 8, Limb, float>;       // a line's coefficient

template <typename Real, int n>
struct LineShape {
  static constexpr int H = n / 2, HE = (n + 1) / 2;          // odd and even parts of a line
  static constexpr int NL = n * n, Np = n * n * n;
  static constexpr int LS = n | 1, PLN = LS * n, PS = PLN * n;   // strides of line, t-plane, population
  static constexpr int M = n - 2, MM = M * M, NI = M * MM, NB = Np - NI;
  static constexpr bool F64 = sizeof(Real) == 8;
  // Populations per work item: about one (FP64: fixed-point accumulators fill the registers) or
  // two (FP32) lines per thread at 256 threads, two tiles of at most about 40 KB.
  static constexpr int PB = F64 ? (n <= 4 ? 14 : n == 5 ? 10 : n == 6 ? 7 : n == 7 ? 5 : n == 8 ? 4 : n == 9 ? 3 : 2)
                                : (n <= 4 ? 27 : n == 5 ? 19 : n == 6 ? 14 : n == 7 ? 10 : n == 8 ? 9 : n == 9 ? 6
                                                                                        : n == 10 ? 5 : n == 11 ? 4 : 3);
  static constexpr int LINES = PB * NL;
  static constexpr int T0 = LINES <= 320 ? LINES : (LINES + 1) / 2;
  static constexpr int T = (T0 + 31) / 32 * 32;
  static constexpr int NPT = (Np + T - 1) / T;               // nodes per thread when gathering
};

// derivative in the even-odd form: d_j = M o + P e, d_{n-1-j} = M o - P e, with
// e_k = v_k + v_{n-1-k}, o_k = v_k - v_{n-1-k} (odd n: e of the middle node is its value)
template <typename Real, int n>
struct StageMats {
  LineCoef<Real> P[LineShape<Real, n>::HE][LineShape<Real, n>::HE];
  LineCoef<Real> M[LineShape<Real, n>::HE][LineShape<Real, n>::HE];
  Real D[sizeof(Real) == 8 ? n * n : 1];    // FP64 fallback of a tile that holds infinities or NaN
  Real w[n];
  int cb;                                    // fixed point: coefficients times 2^cb
  LineCoef<Real> B;                          // stage weight; fixed point: times 2^62
};
// filter v + sum_k g_k U_k (W_k . v) over the modes k >= 2: mode k has the parity of k, so W_k
// reads the even or the odd half of the line and U_k adds to that half (end rows are zero)
template <typename Real, int n>
struct FilterMats {
  LineCoef<Real> U[n][LineShape<Real, n>::HE];
  LineCoef<Real> W[n][LineShape<Real, n>::HE];
  Real Ud[sizeof(Real) == 8 ? n : 1][n], Wd[sizeof(Real) == 8 ? n : 1][n];   // FP64 fallback
  Real g[n];                                 // sigma_k - 1 of the fixed filter
  Real w[n];
  int cw, cu;
  int ex;                                    // biased exponent of the largest |g|
};

template <typename Real, int n, typename Host>
StageMats<Real, n> make_stage_mats(const Host &h) {
  using S = LineShape<Real, n>;
  StageMats<Real, n> m{};
  double P[S::HE][S::HE] = {}, M[S::HE][S::HE] = {}, row = 0;
  for (int j = 0; j < S::HE; ++j) {
    double sum = 0;
    for (int k = 0; k < S::HE; ++k) {
      const double a = h.D[j * n + k], b = h.D[j * n + n - 1 - k];
      const bool cj = 2 * j == n - 1, ck = 2 * k == n - 1;   // middle row and column of odd n
      P[j][k] = cj ? 0.0 : (ck ? a : 0.5 * (a + b));
      M[j][k] = ck ? 0.0 : 0.5 * (a - b);
      sum += std::fabs(P[j][k]) + std::fabs(M[j][k]);
    }
    row = std::max(row, sum);
  }
  for (int k = 0; k < n; ++k) m.w[k] = (Real)h.w[k];
  if constexpr (S::F64) {
    m.cb = fix_shift(row, 62);
    for (int j = 0; j < S::HE; ++j)
      for (int k = 0; k < S::HE; ++k) {
        // halves of sums and differences of the FP64 entries, without the rounding of an FP64 sum
        const long long a = std::llrint(std::ldexp(h.D[j * n + k], m.cb - 1)), b = std::llrint(std::ldexp(h.D[j * n + n - 1 - k], m.cb - 1));
        const bool cj = 2 * j == n - 1, ck = 2 * k == n - 1;
        m.P[j][k] = limbs(cj ? 0 : ck ? 2 * a : a + b);
        m.M[j][k] = limbs(ck ? 0 : a - b);
      }
    for (int k = 0; k < n * n; ++k) m.D[k] = h.D[k];
  } else {
    for (int j = 0; j < S::HE; ++j)
      for (int k = 0; k < S::HE; ++k) { m.P[j][k] = (float)P[j][k]; m.M[j][k] = (float)M[j][k]; }
  }
  return m;
}

template <typename Real, int n, typename Host>
FilterMats<Real, n> make_filter_mats(const Host &h) {
  using S = LineShape<Real, n>;
  FilterMats<Real, n> m{};
  double rw = 0, ru = 0;
  for (int j = 0; j < n; ++j) {
    double su = 0, sw = 0;
    for (int k = 0; k < n; ++k) { su += std::fabs(h.Vm[j * n + k]); sw += std::fabs(h.Vinv[j * n + k]); }
    ru = std::max(ru, su);
    rw = std::max(rw, sw);
  }
  m.cw = fix_shift(rw, 61);
  m.cu = fix_shift(ru, 61);
  for (int k = 0; k < n; ++k) {
    m.g[k] = (Real)(h.fixed_sigma[k] - 1.0);
    if (h.fixed_sigma[k] != 1.0) m.ex = std::max(m.ex, std::max(0, 1023 + std::ilogb(h.fixed_sigma[k] - 1.0)));
    m.w[k] = (Real)h.w[k];
    for (int j = 0; j < S::HE; ++j) {
      const double u = j == 0 || k < 2 ? 0.0 : h.Vm[j * n + k], w = k < 2 ? 0.0 : h.Vinv[k * n + j];
      const bool mid = 2 * j == n - 1;
      if constexpr (S::F64) {
        m.U[k][j] = fix_coef(mid && (k & 1) ? 0.0 : u, m.cu);
        m.W[k][j] = fix_coef(mid && (k & 1) ? 0.0 : w, m.cw);
      } else {
        m.U[k][j] = (float)(mid && (k & 1) ? 0.0 : u);
        m.W[k][j] = (float)(mid && (k & 1) ? 0.0 : w);
      }
    }
    if constexpr (S::F64)
      for (int j = 0; j < n; ++j) {
        m.Ud[k][j] = j == 0 || j == n - 1 || k < 2 ? 0.0 : h.Vm[j * n + k];
        m.Wd[k][j] = k < 2 ? 0.0 : h.Vinv[k * n + j];
      }
  }
  return m;
}

// a term of a derivative: from N = 12 on with the high word of the lowest product.  Error against long
// double, smooth lines at the tile's scale, in units of 2^-57 (row sum)(largest value): N = 7 0.27 (FP64 with
// even and odd parts 1.31), N = 11 0.62 (0.72), N = 14 0.17 (0.69; 0.78 without the high word).
template <int n>
__device__ __forceinline__ void fix_mac_line(Fix128 &s, const Limb &c, const Limb &q) {
  if constexpr (n > 12) fix_mac_full(s, c, q);
  else fix_mac(s, c, q);
}
// d = D v in units of 2^(61 - cb) of v's
template <int n>
__device__ __forceinline__ void line_deriv(const StageMats<double, n> &m, const long long (&v)[n], long long (&d)[n]) {
  constexpr int H = n / 2, HE = (n + 1) / 2;
  Limb e[HE], o[H];
#pragma unroll
  for (int k = 0; k < H; ++k) { e[k] = limbs(v[k] + v[n - 1 - k]); o[k] = limbs(v[k] - v[n - 1 - k]); }
  if constexpr (n & 1) e[H] = limbs(v[H]);
#pragma unroll
  for (int j = 0; j < HE; ++j) {
    Fix128 sm{0, 0}, sp{0, 0};
#pragma unroll
    for (int k = 0; k < H; ++k) fix_mac_line<n>(sm, m.M[j][k], o[k]);
    if (2 * j == n - 1) {
      d[j] = fix_top<3>(sm);
    } else {
#pragma unroll
      for (int k = 0; k < HE; ++k) fix_mac_line<n>(sp, m.P[j][k], e[k]);
      const Fix128 a{sm.A + sp.A, sm.B + sp.B}, b{sm.A - sp.A, sm.B - sp.B};
      d[j] = fix_top<3>(a);
      d[n - 1 - j] = fix_top<3>(b);
    }
  }
}

// |q| < 2^57: a pass grows a tile's largest value by at most 3.8 for transfer functions in [0, 1]
// (N <= 9; N = 14: 5.0), three passes stay below 2^63 and the sums of a pair before the last below 2^62.
constexpr int kFilterShift = 4;
// sigma_k - 1 is taken times 2^(60 + shift): a weak filter's change keeps its bits.  ex: largest exponent
// of |sigma_k - 1| (at most 1)
template <int n>
__host__ __device__ __forceinline__ int filter_up(const FilterMats<double, n> &m) { return 123 - m.cu - m.cw; }
template <int n>
__device__ __forceinline__ int filter_gain_shift(const FilterMats<double, n> &m, int ex) {
  return min(max(1022 - ex, 0), filter_up(m));
}
__device__ __forceinline__ long long filter_gain(double g, int shift) { return __double2ll_rn(scalbn(g, 60 + shift)); }
// v <- v + sum_k g_k U_k (W_k . v), g from filter_gain.  Even modes first: their correction is the same at
// both ends of a pair and leaves the differences that the odd modes read unchanged, so one half's sums are
// in registers at a time (and the even half's fractions).  Rounding: s = W_k . v to a fraction of v's unit
// times g, both halves' corrections together to the nearest unit.
template <int n>
__device__ __forceinline__ void line_filter(const FilterMats<double, n> &m, const long long *g, int shift, long long (&v)[n]) {
  constexpr int H = n / 2, HE = (n + 1) / 2;
  const int up = filter_up(m) - shift;                  // to the units of v
  int fe[HE];                                           // fractions of the even half, in 2^-29
  auto half = [&](auto qc) {
    constexpr int q = decltype(qc)::value, K = q ? H : HE;
    Limb x[K];
#pragma unroll
    for (int j = 0; j < K; ++j) x[j] = limbs(2 * j == n - 1 ? v[j] : (q ? v[j] - v[n - 1 - j] : v[j] + v[n - 1 - j]));
    Fix128 ac[K];
#pragma unroll
    for (int j = 0; j < K; ++j) ac[j] = Fix128{0, 0};
#pragma unroll
    for (int k = 2 + q; k < n; k += 2) {
      const long long gk = g[k];
      if (gk != 0) {
        Fix128 s{0, 1ll << 26}, t{0, 1ll << 27};
#pragma unroll
        for (int j = 0; j < K; ++j) fix_mac_full(s, m.W[k][j], x[j]);
        fix_mac_full(t, limbs(gk), limbs(fix_top<5>(s)));
        const Limb y = limbs(fix_top<4>(t));            // g s in units of 2^(59 - cw - shift)
#pragma unroll
        for (int j = 1; j < K; ++j) fix_mac_full(ac[j], m.U[k][j], y);
      }
    }
#pragma unroll
    for (int j = 1; j < K; ++j) {
      const long long a = (long long)((unsigned long long)ac[j].A << up) + (ac[j].B >> (32 - up));
      const int f = (int)(((unsigned)ac[j].B << up) >> 3);
      if constexpr (q == 0) {
        fe[j] = f;
        v[j] += a;
        if (2 * j != n - 1) v[n - 1 - j] += a;
      } else {
        v[j] += a + ((fe[j] + f + (1 << 28)) >> 29);
        v[n - 1 - j] += ((fe[j] - f + (1 << 28)) >> 29) - a;
      }
    }
    if constexpr (q == 1 && (n & 1)) v[H] += (fe[H] + (1 << 28)) >> 29;
  };
  half(std::integral_constant<int, 0>{});
  half(std::integral_constant<int, 1>{});
}

}  // namespace slb
