// Population-split element kernels for hexahedra at any order: one CTA per (element, group of
// populations), one thread per line of a pass.
//
//   lines_stage_kernel   advection stage: -B dt e.grad f by sum factorisation (r-, s-, t-pass),
//                        flux bounce-back, stage combination of element-interior nodes, weighted
//                        shares of element-boundary nodes to the assembly trace
//   lines_filter_kernel  explicit filter I + U W along r, s and t, the transfer function fixed or
//                        chosen per element
//
// Once collided, a population advects and filters on its own, so a group of any size is a work
// item and the lattice enters only through run-time velocity masks: one instantiation per order,
// precision and element kind serves both lattices.  Every pass forms its line products in the
// even-odd form (the GLL nodes are symmetric, so derivative and filter map even parts to odd or
// even parts: half the multiply-adds).  FP32 lines are FP32; FP64 lines are 64-bit fixed point
// (selbm_fixed_lines.cuh), since two FP64 operations per clock and SM bound everything else.  FP64,
// Taylor-Green 16^3, N = 7, D3Q27: a stage 798 us (2.59 ms in FP64 arithmetic), integer multiply-adds at 53 %
// and issue at 51 % of their peaks with 35 % of the warps (80 registers and 41 KB: three CTAs); the filter
// 632 us, ALU 61 %.
//
// The t-pass comes last and writes global memory itself: lanes run over (i0, i1), so a store of
// one t-index is as coalesced as a node-ordered copy, and f^0, the wall-free result and the share
// never return to shared memory.  Element-interior nodes are numbered first, element by element
// in local order, so their addresses need no index.  Lines in shared memory are padded to an odd
// stride (no bank conflicts along r).
#pragma once
#include <cuda_runtime.h>

#include <algorithm>
#include <type_traits>
#include <vector>

#include "selbm_collide.cuh"
#include "selbm_fixed_lines.cuh"
#include "selbm_kernels.cuh"
#include "selbm_lines.h"
#include "selbm_smem.cuh"
#include "selbm_split_stage.cuh"

namespace slb {

template <int LAT>
LatticeRT lattice_rt() {
  constexpr VelTab V = LT<LAT>::v;
  LatticeRT l{};
  l.Q = V.Q;
  for (int k = 0; k < 3; ++k) { l.pos[k] = vel_mask(V, k, 1); l.neg[k] = vel_mask(V, k, -1); }
  for (int a = 0; a < V.Q; ++a) { l.td[a] = V.t[a]; l.tf[a] = (float)V.t[a]; l.opp[a] = (signed char)V.opp[a]; }
  return l;
}

// ---------------------------------------------------------------------------
// line operations
// ---------------------------------------------------------------------------
// d = D v
template <int n>
__device__ __forceinline__ void line_deriv(const StageMats<float, n> &m, const float (&v)[n], float (&d)[n]) {
  constexpr int H = n / 2, HE = (n + 1) / 2;
  float2 eo[HE];
#pragma unroll
  for (int k = 0; k < H; ++k) eo[k] = make_float2(v[k] + v[n - 1 - k], v[k] - v[n - 1 - k]);
  if constexpr (n & 1) eo[H] = make_float2(v[H], 0.f);
#pragma unroll
  for (int j = 0; j < HE; ++j) {
    float2 s = __fmul2_rn(make_float2(m.P[j][0], m.M[j][0]), eo[0]);
#pragma unroll
    for (int k = 1; k < HE; ++k) s = __ffma2_rn(make_float2(m.P[j][k], m.M[j][k]), eo[k], s);
    if (2 * j == n - 1) d[j] = s.y;
    else { d[j] = s.y + s.x; d[n - 1 - j] = s.y - s.x; }
  }
}
// v <- v + sum_k g_k U_k (W_k . v)
template <int n>
__device__ __forceinline__ void line_filter(const FilterMats<float, n> &m, const float *g, float (&v)[n]) {
  constexpr int H = n / 2, HE = (n + 1) / 2;
  float eo[2][HE], ac[2][HE];
#pragma unroll
  for (int k = 0; k < H; ++k) { eo[0][k] = v[k] + v[n - 1 - k]; eo[1][k] = v[k] - v[n - 1 - k]; }
  if constexpr (n & 1) { eo[0][H] = v[H]; eo[1][H] = 0.f; }
#pragma unroll
  for (int j = 0; j < HE; ++j) { ac[0][j] = 0.f; ac[1][j] = 0.f; }
#pragma unroll
  for (int k = 2; k < n; ++k) {
    const float gk = g[k];
    if (gk != 0.f) {
      const int q = k & 1;
      float s = 0.f;
#pragma unroll
      for (int j = 0; j < (q ? H : HE); ++j) s += m.W[k][j] * eo[q][j];
      s *= gk;
#pragma unroll
      for (int j = 1; j < (q ? H : HE); ++j) ac[q][j] += m.U[k][j] * s;
    }
  }
#pragma unroll
  for (int j = 1; j < H; ++j) { v[j] += ac[0][j] + ac[1][j]; v[n - 1 - j] += ac[0][j] - ac[1][j]; }
  if constexpr (n & 1) v[H] += ac[0][H];
}
// ---------------------------------------------------------------------------
// gather of one group's tile
// ---------------------------------------------------------------------------
template <typename Real, int n>
__device__ __forceinline__ int tile_offset(int i) {
  using S = LineShape<Real, n>;
  const int i0 = i % n, i1 = (i / n) % n, i2 = i / (n * n);
  return i0 + S::LS * i1 + S::PLN * i2;
}
// tile[pl][node] of populations a0 .. a0 + na - 1; FP64: fixed point at the population's largest
// exponent em[pl] (2047: the tile holds infinities or NaN and keeps its FP64 values).  Ends with
// the tile visible to the CTA.
template <typename Real, int n, int SHIFT>
__device__ __forceinline__ void gather_lines(LineVal<Real> *tile, int *em, const Real *fin, size_t G, const int32_t *l2g,
                                             int na, int tid) {
  using S = LineShape<Real, n>;
  if constexpr (!S::F64) {
    const unsigned s0 = (unsigned)__cvta_generic_to_shared(tile);
#pragma unroll
    for (int r = 0; r < S::NPT; ++r) {
      const int i = tid + r * S::T;
      if (i < S::Np) {
        const float *src = fin + l2g[i];
        const unsigned d = s0 + 4u * (unsigned)tile_offset<Real, n>(i);
#pragma unroll 4
        for (int pl = 0; pl < na; ++pl) cp_async_s<float>(d + pl * S::PS * 4u, src + (size_t)pl * G);
      }
    }
    cp_async_wait_all();
    __syncthreads();
  } else {
    double raw[S::NPT][S::PB];
#pragma unroll
    for (int r = 0; r < S::NPT; ++r) {
      const int i = tid + r * S::T;
      const double *src = fin + (i < S::Np ? l2g[i] : 0);
#pragma unroll
      for (int pl = 0; pl < S::PB; ++pl) raw[r][pl] = (i < S::Np && pl < na) ? __ldg(src + (size_t)pl * G) : 0.0;
    }
#pragma unroll
    for (int pl = 0; pl < S::PB; ++pl) {
      int e = kMinExp;
#pragma unroll
      for (int r = 0; r < S::NPT; ++r) e = max(e, exp_of(raw[r][pl]));
      e = __reduce_max_sync(0xffffffffu, e);
      if (pl < na && (tid & 31) == 0) atomicMax(&em[pl], e);
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < S::NPT; ++r) {
      const int i = tid + r * S::T;
      if (i < S::Np) {
        const int o = tile_offset<Real, n>(i);
#pragma unroll
        for (int pl = 0; pl < S::PB; ++pl)
          if (pl < na) {
            const int ex = em[pl];
            tile[pl * S::PS + o] =
                ex == 2047 ? __double_as_longlong(raw[r][pl]) : to_fixed<SHIFT>(raw[r][pl], ex);
          }
      }
    }
    __syncthreads();
  }
}

// base offset and stride of line L along an axis
template <typename Real, int n, int AX>
__device__ __forceinline__ int line_base(int L) {
  using S = LineShape<Real, n>;
  if constexpr (AX == 0) return S::LS * (L % n) + S::PLN * (L / n);
  else if constexpr (AX == 1) return (L % n) + S::PLN * (L / n);
  else return (L % n) + S::LS * (L / n);
}
template <typename Real, int n, int AX>
constexpr int line_stride() {
  using S = LineShape<Real, n>;
  return AX == 0 ? 1 : (AX == 1 ? S::LS : S::PLN);
}

// FP64 line derivative of a tile that holds infinities or NaN: FP64 arithmetic, one node at a time
template <int n>
__device__ __noinline__ double slow_deriv(const double *D, const long long *row, int stride, int j) {
  double s = 0;
#pragma unroll 1
  for (int k = 0; k < n; ++k) s += D[j * n + k] * __longlong_as_double(row[k * stride]);
  return s;
}

// ---------------------------------------------------------------------------
// advection stage
// ---------------------------------------------------------------------------
constexpr int kMetricShift = 5;
template <typename Real, int n, bool AFFINE>
constexpr size_t lines_stage_smem(int pb, int wall_max) {
  using S = LineShape<Real, n>;
  size_t b = (size_t)(2 * pb + (AFFINE ? 0 : 3)) * S::PS * sizeof(LineVal<Real>);   // tile, sums, metrics of one axis
  b += (size_t)pb * 3 * sizeof(LineVal<Real>);                                      // coefficients of the axes
  b += (size_t)(2 * pb + (size_t)pb * wall_max) * sizeof(Real);                     // force, wall terms
  if (S::F64 && AFFINE) b += (size_t)S::Np * sizeof(double);                        // quadrature weights
  return b + (size_t)3 * pb * sizeof(int) + 16;
}

template <typename Real, int n, bool AFFINE>
__global__ void __launch_bounds__(LineShape<Real, n>::T, LineShape<Real, n>::F64 ? 3 : (n <= 8 ? 5 : 3))
lines_stage_kernel(const KParams<Real> p, const StageMats<Real, n> m, const LatticeRT lt, const LineGeo<Real> lg,
                   const int pb, const int ng) {
  using S = LineShape<Real, n>;
  using Val = LineVal<Real>;
  constexpr int NL = S::NL, PS = S::PS, T = S::T, Np = S::Np;
  constexpr int SHIFT = FixScale<n>::SHIFT;
  constexpr bool F64 = S::F64;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Val *tile = reinterpret_cast<Val *>(smem_raw);      // [pb][PS] f^{s-1}
  Val *acc = tile + pb * PS;                           // [pb][PS] sums of the passes
  Val *sg = acc + pb * PS;                             // curved: [3][PS] dr_l/dx_k of the axis in hand
  Val *cf = sg + (AFFINE ? 0 : 3 * PS);                // [pb][3] affine: -B dt sum_k e_k dr_l/dx_k
  Real *fc = reinterpret_cast<Real *>(cf + pb * 3);    // [2][pb] B dt F*_a / rho; B dt 3 t_a
  Real *wbuf = fc + 2 * pb;                            // [wall nodes][pb]
  Real *sw = wbuf + (size_t)pb * p.wall_max;           // FP64, affine: [Np] J w w w
  int *em = reinterpret_cast<int *>(sw + (F64 && AFFINE ? Np : 0));   // [pb] exponent of the tile
  int *ge = em + pb;                                   // [pb] exponent of the coefficients
  int *axes = ge + pb;                                 // [pb] bit l: the axis has a coefficient
  const int e = blockIdx.x / ng, a0 = (blockIdx.x - e * ng) * pb;
  const int na = min(pb, lt.Q - a0);
  const int tid = threadIdx.x;
  const Real Bdt = p.B * p.dt;
  const int32_t *l2g = p.l2g + (size_t)e * Np;
  const size_t G = p.Gs;
  auto sgn = [&](int k, int a) -> int { return (int)((lt.pos[k] >> a) & 1u) - (int)((lt.neg[k] >> a) & 1u); };

  if (F64 && tid < pb) em[tid] = kMinExp;
  if (tid < na) {
    int on = 0;
    if constexpr (AFFINE && F64) {
      // -dt sum_k e_k dr_l/dx_k in fixed point from the table, times B
      const size_t row = (size_t)e * lt.Q + a0 + tid;
      ge[tid] = lg.gexp[row];
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        const long long c = lg.g[row * 3 + l];
        Fix128 t{0, 1ll << 29};
        fix_mac(t, m.B, limbs(c));
        cf[tid * 3 + l] = fix_top<2>(t);
        on |= (c != 0) << l;
      }
    } else if constexpr (AFFINE) {
#pragma unroll
      for (int l = 0; l < 3; ++l) {
        Real c = 0;
#pragma unroll
        for (int k = 0; k < 3; ++k) c += Real(sgn(k, a0 + tid)) * p.el_drdx[((size_t)e * 3 + l) * 3 + k];
        cf[tid * 3 + l] = -Bdt * c;
        on |= (c != Real(0)) << l;
      }
    } else {
      on = ((lt.pos[0] | lt.neg[0] | lt.pos[1] | lt.neg[1] | lt.pos[2] | lt.neg[2]) >> (a0 + tid)) & 1u ? 7 : 0;
    }
    axes[tid] = on;
  }
  if (p.has_force && tid < na) {
    Real g3 = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) g3 += Real(sgn(k, a0 + tid)) * p.g[k];
    const Real ta = lt.t<Real>(a0 + tid);
    fc[tid] = Bdt * ta * Real(3) * g3;
    fc[pb + tid] = Bdt * ta * Real(3);
  }
  if constexpr (F64 && AFFINE) {
    const double J = p.el_J[e];
    for (int i = tid; i < Np; i += T) sw[i] = J * lg.w3[i];
  }
  if (F64) __syncthreads();                            // em
  gather_lines<Real, n, SHIFT>(tile, em, p.fin + (size_t)a0 * G, G, l2g, na, tid);

  // metrics of one axis (curved elements)
  auto stage_metrics = [&](int l) {
    if constexpr (!AFFINE) {
      __syncthreads();
      const Real *src = p.drdx + ((size_t)e * 9 + 3 * l) * Np;
      const int top = F64 ? lg.gexp[e] : 0;
      for (int i = tid; i < Np; i += T) {
        const int o = tile_offset<Real, n>(i);
#pragma unroll
        for (int k = 0; k < 3; ++k) {
          const Real v = __ldg(src + (size_t)k * Np + i);
          // fixed point: magnitudes below 2^58, three of them below 2^60
          if constexpr (F64) sg[k * PS + o] = to_fixed_rn<kMetricShift>(v, top);
          else sg[k * PS + o] = v;
        }
      }
      __syncthreads();
    }
  };
  // c_l (D_l f) of one line, added to in[] (nothing where the coefficient vanishes)
  auto line_terms = [&](auto axc, int pl, int base, Val (&in)[n]) {
    constexpr int AX = decltype(axc)::value;
    constexpr int ST = line_stride<Real, n, AX>();
    const int a = a0 + pl;
    const Val *row = tile + pl * PS + base;
    Val v[n], d[n];
#pragma unroll
    for (int k = 0; k < n; ++k) v[k] = row[k * ST];
    line_deriv<n>(m, v, d);
    if constexpr (AFFINE) {
      if constexpr (F64) {
        const Limb c = limbs(cf[pl * 3 + AX]);
#pragma unroll
        for (int j = 0; j < n; ++j) {
          Fix128 t{0, 0};
          fix_mac(t, c, limbs(d[j]));
          in[j] += fix_top<0>(t);
        }
      } else {
        const float c = cf[pl * 3 + AX];
#pragma unroll
        for (int j = 0; j < n; ++j) in[j] += c * d[j];
      }
    } else {
      const int e0 = sgn(0, a), e1 = sgn(1, a), e2 = sgn(2, a);
      const Val *gm = sg + base;
#pragma unroll
      for (int j = 0; j < n; ++j) {
        const Val c = (Val)e0 * gm[j * ST] + (Val)e1 * gm[PS + j * ST] + (Val)e2 * gm[2 * PS + j * ST];
        if constexpr (F64) {
          Fix128 t{0, 0};
          fix_mac(t, limbs(c), limbs(d[j]));
          in[j] += fix_top<0>(t);
        } else {
          in[j] += c * d[j];
        }
      }
    }
  };
  // the same in FP64 for a tile with infinities or NaN, node j of the line
  auto slow_term = [&](int ax, int pl, int base, int st, int j) -> double {
    if constexpr (F64) {
      double c = 0;
      if (AFFINE) {
        c = from_fixed(cf[pl * 3 + ax], -ge[pl]);
        if (c == 0) return 0.0;
      } else {
        const int off = base + j * st;
        const int i = off % S::LS + n * ((off / S::LS) % n) + n * n * (off / S::PLN);
        const double *gm = p.drdx + ((size_t)e * 9 + 3 * ax) * Np + i;
        for (int k = 0; k < 3; ++k) c += sgn(k, a0 + pl) * gm[k * Np];
      }
      return c * slow_deriv<n>(m.D, tile + pl * PS + base, st, j);
    } else return 0.0;
  };
  // ---- r-pass: sums start; s-pass: sums grow
  stage_metrics(0);
  for (int t = tid; t < na * NL; t += T) {
    const int pl = t / NL, base = line_base<Real, n, 0>(t - pl * NL);
    if (!(axes[pl] & 1)) continue;
    Val *dst = acc + pl * PS + base;
    if (F64 && em[pl] == 2047) {
      if constexpr (F64)
        for (int j = 0; j < n; ++j) dst[j] = __double_as_longlong(slow_term(0, pl, base, 1, j));
      continue;
    }
    Val s[n];
#pragma unroll
    for (int j = 0; j < n; ++j) s[j] = 0;
    line_terms(std::integral_constant<int, 0>{}, pl, base, s);
#pragma unroll
    for (int j = 0; j < n; ++j) dst[j] = s[j];
  }
  stage_metrics(1);
  if (AFFINE) __syncthreads();
  for (int t = tid; t < na * NL; t += T) {
    const int pl = t / NL, base = line_base<Real, n, 1>(t - pl * NL);
    const int on = axes[pl];
    if (!(on & 2)) continue;
    constexpr int ST = line_stride<Real, n, 1>();
    Val *dst = acc + pl * PS + base;
    const bool more = on & 1;
    if (F64 && em[pl] == 2047) {
      if constexpr (F64)
        for (int j = 0; j < n; ++j)
          dst[j * ST] = __double_as_longlong((more ? __longlong_as_double(dst[j * ST]) : 0.0) + slow_term(1, pl, base, ST, j));
      continue;
    }
    Val s[n];
#pragma unroll
    for (int j = 0; j < n; ++j) s[j] = more ? dst[j * ST] : Val(0);
    line_terms(std::integral_constant<int, 1>{}, pl, base, s);
#pragma unroll
    for (int j = 0; j < n; ++j) dst[j * ST] = s[j];
  }

  // ---- flux bounce-back terms of the group's populations at this element's wall nodes
  //      (Sec. 2.2.1), from the unique-node array
  const int w0 = p.wall_off[e], nw = p.wall_off[e + 1] - w0;
  for (int idx = tid; idx < na * nw; idx += T) {
    const int k = idx / na, pl = idx - k * na, a = a0 + pl;
    const WallPt<Real> &wp = p.walls[w0 + k];
    const size_t g = l2g[wp.i];
    const Real diff = p.fin[(size_t)a * G + g] - p.fin[(size_t)lt.opp[a] * G + g];
    const Real t6 = Real(2) * lt.t<Real>(a) * p.rho0 * Real(3);
    Real sum = 0;
    for (int f = 0; f < wp.nf; ++f) {
      Real ne = 0, eu = 0;
      const Real *ub = p.wall_u + 3 * (wp.wid[f] - 1);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const Real s = Real(sgn(c, a));
        ne += s * wp.n[f][c];
        eu += s * ub[c];
      }
      if (ne < Real(0)) sum += wp.wsJs[f] * ne * (diff - t6 * eu);
    }
    wbuf[k * pb + pl] = Bdt * sum;
  }

  // ---- t-pass, stage combination and output
  stage_metrics(2);
  if (AFFINE) __syncthreads();
  const size_t EN = (size_t)p.E * S::NB;
  const bool use_f0 = p.stage != 1;
  for (int t = tid; t < na * NL; t += T) {
    const int pl = t / NL, L = t - pl * NL, a = a0 + pl;
    const int base = line_base<Real, n, 2>(L), i0 = L % n, i1 = L / n;
    constexpr int ST = line_stride<Real, n, 2>();
    const int on = axes[pl];
    const bool more = on & 3;
    const bool slow = F64 && em[pl] == 2047;
    const bool lin = i0 > 0 && i0 < n - 1 && i1 > 0 && i1 < n - 1;
    // interior lines read f^0 (and f^{s-1}) and write f^s, edge lines write their shares: node k of the
    // middle planes is `step` values after node k - 1 in either, so one code path serves both
    const size_t gi = (size_t)a * G + (size_t)e * S::NI + (lin ? (i0 - 1) + S::M * (i1 - 1) : 0);   // node k: + MM (k - 1)
    Real f0v[S::M], fv[S::M];
#pragma unroll
    for (int k = 0; k < S::M; ++k) {
      f0v[k] = lin && use_f0 ? __ldg(p.f0 + gi + (size_t)(S::MM * k)) : Real(0);
      if constexpr (F64) fv[k] = lin ? __ldg(p.fin + gi + (size_t)(S::MM * k)) : Real(0);
      else fv[k] = lin ? tile[pl * PS + base + (k + 1) * ST] : Real(0);
    }
    Val s[n];
    const Val *ac = acc + pl * PS + base;
    if (!slow) {
#pragma unroll
      for (int j = 0; j < n; ++j) s[j] = more ? ac[j * ST] : Val(0);
      if (on & 4) line_terms(std::integral_constant<int, 2>{}, pl, base, s);
    } else if constexpr (F64) {
#pragma unroll
      for (int j = 0; j < n; ++j)
        s[j] = __double_as_longlong((more ? __longlong_as_double(ac[j * ST]) : 0.0) + (on & 4 ? slow_term(2, pl, base, ST, j) : 0.0));
    }
    // value of a sum: curved elements carry -B dt here
    int ex = 0;
    if constexpr (F64) {
      const int gs = AFFINE ? ge[pl] : 1023 + 52 + kMetricShift - lg.gexp[e];
      ex = 125 - gs - m.cb + em[pl] - FixScale<n>::EXP0;
    }
    auto value = [&](Val x) -> Real {
      if constexpr (F64) return slow ? __longlong_as_double(x) : from_fixed(x, ex);
      else return x;
    };
    const Real scale = AFFINE ? Real(1) : -Bdt;
    const Real w01 = AFFINE && !F64 ? p.el_J[e] * m.w[i0] * m.w[i1] : Real(0);
    auto share_weight = [&](int k) -> Real {
      if constexpr (!AFFINE) return scale * p.wJ[(size_t)e * Np + L + k * NL];
      else if constexpr (F64) return sw[L + k * NL];
      else return w01 * m.w[k];
    };
    // boundary slots: nodes before this one, less the interior ones among them
    const int before = min(max(i1 - 1, 0), S::M) * S::M + (i1 >= 1 && i1 <= S::M ? min(max(i0 - 1, 0), S::M) : 0);
    Real *tp = p.T + (size_t)a * EN + (size_t)e * S::NB + L;
    tp[0] = share_weight(0) * value(s[0]);
    tp[(n - 1) * NL - S::NI] = share_weight(n - 1) * value(s[n - 1]);
    Real *dst = lin ? p.fout + gi : tp + NL - before;
    const int step = lin ? S::MM : NL - S::MM;
    const Real Bl = lin ? p.B : Real(0), Al = lin && use_f0 ? p.A : Real(0);
    if (!p.has_force) {
#pragma unroll
      for (int k = 1; k < n - 1; ++k) {
        const Real x = value(s[k]);
        Real c = scale;
        if (!lin) c = share_weight(k);
        Real out = (AFFINE && F64 && lin) ? Bl * fv[k - 1] + x : Bl * fv[k - 1] + c * x;
        if (!F64 || (lin && use_f0)) out += Al * f0v[k - 1];
        *dst = out;
        dst += step;
      }
    } else {
      const Real famp = p.fS ? *p.famp : Real(0);
#pragma unroll 1
      for (int k = 1; k < n - 1; ++k) {
        Real fk = 0, f0k = 0;
        Val sk = 0;
#pragma unroll
        for (int q = 1; q < n - 1; ++q)
          if (q == k) { sk = s[q]; fk = fv[q - 1]; f0k = f0v[q - 1]; }
        const Real x = value(sk);
        if (lin) {
          Real out = Bl * fk + scale * x + Al * f0k;
          const size_t g = (size_t)e * S::NI + (i0 - 1) + S::M * ((i1 - 1) + S::M * (k - 1));
          Real fa = fc[pl];
          if (p.fS) {
            Real es = 0;
#pragma unroll
            for (int c = 0; c < 3; ++c) es += Real(sgn(c, a)) * p.fS[(size_t)c * p.G + g];
            fa += fc[pb + pl] * famp * es;
          }
          *dst = out + fa * p.rho[g];
        } else {
          *dst = share_weight(k) * x;
        }
        dst += step;
      }
    }
  }
  if (nw > 0) {
    // wall terms join the weighted shares of their boundary nodes
    __syncthreads();
    for (int idx = tid; idx < na * nw; idx += T) {
      const int k = idx / na, pl = idx - k * na;
      p.T[(size_t)(a0 + pl) * EN + (size_t)e * S::NB + p.walls[w0 + k].b] += wbuf[k * pb + pl];
    }
  }
}

// ---------------------------------------------------------------------------
// explicit filter
// ---------------------------------------------------------------------------
template <typename Real, int n>
constexpr size_t lines_filter_smem(int pb) {
  using S = LineShape<Real, n>;
  return (size_t)pb * S::PS * sizeof(LineVal<Real>) + n * (sizeof(LineVal<Real>) + sizeof(Real)) + pb * sizeof(int) + 16;
}

// LEARNED: the element's transfer function sigma[e][n]; element-interior nodes to out, weighted
// shares wJ f of boundary nodes to the trace.  Otherwise the fixed filter; every node is written
// by its owner (the copies agree).  Writing the integers back instead of the value plus the tile's change
// would take 588 us instead of 632 (FP64, as above), and the low bits of values small next to the tile's largest.
template <typename Real, int n, bool LEARNED>
__global__ void __launch_bounds__(LineShape<Real, n>::T, LineShape<Real, n>::F64 ? 3 : (n <= 8 ? 5 : 3))
lines_filter_kernel(const KParams<Real> p, const FilterMats<Real, n> m, const Real *sigma, Real *out, const int Q,
                    const int pb, const int ng) {
  using S = LineShape<Real, n>;
  using Val = LineVal<Real>;
  constexpr int NL = S::NL, PS = S::PS, T = S::T, Np = S::Np;
  constexpr bool F64 = S::F64;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Val *tile = reinterpret_cast<Val *>(smem_raw);            // [pb][PS]
  Val *sgk = tile + pb * PS;                                 // [n] sigma_k - 1
  Real *sgd = reinterpret_cast<Real *>(sgk + n);             // [n] the same as a Real
  int *em = reinterpret_cast<int *>(sgd + n);                // [pb]
  int *gsh = em + pb;                                        // FP64: shift of sgk (filter_gain)
  const int e = blockIdx.x / ng, a0 = (blockIdx.x - e * ng) * pb;
  const int na = min(pb, Q - a0);
  const int tid = threadIdx.x;
  const int32_t *l2g = p.l2g + (size_t)e * Np;
  const size_t G = p.Gs;
  if (F64 && tid < pb) em[tid] = kMinExp;
  if (tid < 32) {
    const int k = min(tid, n - 1);
    const Real g = LEARNED ? sigma[(size_t)e * n + k] - Real(1) : m.g[k];
    Val gk;
    if constexpr (F64) {
      const int sh = filter_gain_shift(m, LEARNED ? __reduce_max_sync(0xffffffffu, exp_of(g)) : m.ex);
      gk = filter_gain(g, sh);
      if (tid == 0) *gsh = sh;
    } else gk = g;
    if (tid < n) { sgd[tid] = g; sgk[tid] = gk; }
  }
  if (F64) __syncthreads();
  gather_lines<Real, n, kFilterShift>(tile, em, p.fin + (size_t)a0 * G, G, l2g, na, tid);
  auto filter_line = [&](int pl, Val (&v)[n]) {
    if (F64 && em[pl] == 2047) {
      if constexpr (F64) {
        double o[n];
#pragma unroll
        for (int j = 0; j < n; ++j) o[j] = __longlong_as_double(v[j]);
#pragma unroll 1
        for (int k = 2; k < n; ++k) {
          const double g = sgd[k];
          if (g == 0) continue;
          double s = 0;
#pragma unroll
          for (int j = 0; j < n; ++j) s += m.Wd[k][j] * __longlong_as_double(v[j]);
#pragma unroll
          for (int j = 1; j < n - 1; ++j) o[j] += m.Ud[k][j] * (g * s);
        }
#pragma unroll
        for (int j = 0; j < n; ++j) v[j] = __double_as_longlong(o[j]);
      }
    } else if constexpr (F64) {
      line_filter<n>(m, sgk, *gsh, v);
    } else {
      line_filter<n>(m, sgk, v);
    }
  };
  auto pass = [&](auto axc) {
    constexpr int AX = decltype(axc)::value;
    constexpr int ST = line_stride<Real, n, AX>();
    for (int t = tid; t < na * NL; t += T) {
      const int pl = t / NL;
      Val *row = tile + pl * PS + line_base<Real, n, AX>(t - pl * NL);
      Val v[n];
#pragma unroll
      for (int k = 0; k < n; ++k) v[k] = row[k * ST];
      filter_line(pl, v);
#pragma unroll
      for (int k = 1; k < n - 1; ++k) row[k * ST] = v[k];       // the end values stay as they are
    }
    __syncthreads();
  };
  pass(std::integral_constant<int, 0>{});
  pass(std::integral_constant<int, 1>{});
  pass(std::integral_constant<int, 2>{});
  // one node per thread: its destination is looked up once for the group
  const size_t EN = (size_t)p.E * S::NB;
#pragma unroll 1
  for (int i = tid; i < Np; i += T) {
    const Val *v = tile + tile_offset<Real, n>(i);
    const Real *src = p.fin + (size_t)a0 * G + l2g[i];
    // FP64: the value that came in plus the tile's change, so that neither small values nor modes that
    // stay lose bits to the tile's scale (the loop over the group is unrolled: its loads go out together)
    auto value = [&](int pl) -> Real {
      if constexpr (F64) {
        const int ex = em[pl];
        if (ex == 2047) return __longlong_as_double(v[pl * PS]);
        const double in = __ldg(src + (size_t)pl * G);
        return in + from_fixed(v[pl * PS] - to_fixed<kFilterShift>(in, ex), ex - (1023 + 52 + kFilterShift));
      } else return v[pl * PS];
    };
    Real w = 1;
    Real *dst;
    size_t stride = G;
    if (LEARNED) {
      const int b = p.bslot[i];
      if (b >= 0) {
        w = p.wJ ? p.wJ[(size_t)e * Np + i] : p.el_J[e] * m.w[i % n] * m.w[(i / n) % n] * m.w[i / (n * n)];
        dst = p.T + (size_t)a0 * EN + (size_t)e * S::NB + b;
        stride = EN;
      } else dst = out + (size_t)a0 * G + l2g[i];
    } else {
      if (!p.owner[(size_t)e * Np + i]) continue;
      dst = out + (size_t)a0 * G + l2g[i];
    }
#pragma unroll
    for (int pl = 0; pl < S::PB; ++pl)
      if (pl < na) {
        *dst = LEARNED ? w * value(pl) : value(pl);
        dst += stride;
      }
  }
}

// ---------------------------------------------------------------------------
// launchers
// ---------------------------------------------------------------------------
// Q populations in ng groups of pb, as even as they come
template <typename Real, int n>
void line_groups(int Q, int *pb, int *ng) {
  *ng = (Q + LineShape<Real, n>::PB - 1) / LineShape<Real, n>::PB;
  *pb = (Q + *ng - 1) / *ng;
}

template <typename Real, int n>
cudaError_t launch_lines_stage_t(bool affine, const KParams<Real> &p, const SplitHost &h, const LatticeRT &lt,
                                 const LineGeo<Real> &lg, cudaStream_t s) {
  int pb, ng;
  line_groups<Real, n>(lt.Q, &pb, &ng);
  StageMats<Real, n> m = make_stage_mats<Real, n>(h);
  if constexpr (sizeof(Real) == 8) m.B = fix_coef(p.B, 62);
  else m.B = p.B;
  auto go = [&](auto ac) -> cudaError_t {
    constexpr bool AFFINE = decltype(ac)::value;
    const size_t smem = lines_stage_smem<Real, n, AFFINE>(pb, p.wall_max);
    const cudaError_t err = raise_smem<lines_stage_kernel<Real, n, AFFINE>>(smem);
    if (err != cudaSuccess) return err;
    lines_stage_kernel<Real, n, AFFINE><<<p.E * ng, LineShape<Real, n>::T, smem, s>>>(p, m, lt, lg, pb, ng);
    return cudaGetLastError();
  };
  return affine ? go(std::true_type{}) : go(std::false_type{});
}

template <typename Real, int n>
cudaError_t launch_lines_filter_t(const KParams<Real> &p, const SplitHost &h, int Q, const Real *sigma, Real *out,
                                  cudaStream_t s) {
  int pb, ng;
  line_groups<Real, n>(Q, &pb, &ng);
  const FilterMats<Real, n> m = make_filter_mats<Real, n>(h);
  const size_t smem = lines_filter_smem<Real, n>(pb);
  auto go = [&](auto lc) -> cudaError_t {
    constexpr bool LEARNED = decltype(lc)::value;
    const cudaError_t err = raise_smem<lines_filter_kernel<Real, n, LEARNED>>(smem);
    if (err != cudaSuccess) return err;
    lines_filter_kernel<Real, n, LEARNED><<<p.E * ng, LineShape<Real, n>::T, smem, s>>>(p, m, sigma, out, Q, pb, ng);
    return cudaGetLastError();
  };
  return sigma ? go(std::true_type{}) : go(std::false_type{});
}

// translation units by order: part 0 N <= 6, part 1 above
template <typename Real, int PART>
cudaError_t lines_stage_part(int N, bool affine, const KParams<Real> &p, const SplitHost &h, const LatticeRT &lt,
                             const LineGeo<Real> &lg, cudaStream_t s);
template <typename Real, int PART>
cudaError_t lines_filter_part(int N, const KParams<Real> &p, const SplitHost &h, int Q, const Real *sigma, Real *out,
                              cudaStream_t s);

}  // namespace slb
