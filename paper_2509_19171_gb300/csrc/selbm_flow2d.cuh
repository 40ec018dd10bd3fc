// Resident step of quadrilateral meshes (D2Q9): one cooperative launch runs any number of steps.
//
// A 2D mesh of the method is small: a few MB of state, microseconds of work per step.  As six
// kernels a step its time was launches, gaps and dependent loads (Couette, 32 quads: 74 us a step,
// 82,944-node shear layer: 41 us).  Here every CTA keeps its elements' populations in shared memory
// through all steps: collision, filter and the stages' line products read and write shared memory
// alone, and only the weighted shares of element-boundary nodes cross CTAs, through L2: every 32 bits
// of a share travel in one 8-byte store together with the number of the exchange, and its readers
// poll the share itself.  No flag, fence or grid barrier stands between a store and its reader (a
// release store and acquire polls of the neighbours' flags, the form before, cost about 2 us a
// stage).  Two sets of shares alternate: a CTA that has read its neighbours' shares of exchange k+1
// knows that they have read its own of exchange k.  Copies of a shared node are summed by every CTA
// that holds one, in ascending (element, node) order, so that all copies hold the same bits.
//
// Waits are bounded: a wait that gives up sets *abort (host memory), and every CTA
// leaves; some may have written their share of the state, so it has to be set anew.
#pragma once
#include <cuda_runtime.h>

#include "selbm_flow2d.h"
#include "selbm_lines.cuh"
#include "selbm_moments.cuh"

namespace slb {

// polls of one wait, below a microsecond each.  A constant: with a limit from the launch's arguments, in any
// form of the loop, the FP32 shear layer (32 x 32, N = 8) takes 1.35 instead of 1.15 ms a pass.
constexpr int kFlowSpins = 4000000;
// (population, node) tasks of a CTA up to which FP64 takes a thread per node and not per line.  Few tasks
// leave threads idle in lines, many repeat the line's products.  us a step, node / line: 576 tasks (N = 7, one
// element) 21.1 / 23.4, 1296 (N = 11, one) 34.2 / 42.2, 2187 (N = 8, three) 45.8 / 46.9, 2304 (N = 7, four)
// 53.2 / 51.1, 2592 (N = 11, two) 56.7 / 60.7, 2916 (N = 8, four) 57.9 / 56.9, 3456 (N = 7, six) 74.3 / 68.4,
// 3888 (N = 11, three) 80.9 / 82.2, 4050 (N = 14, two) 85.7 / 89.3: the line lies where neither side loses
// more than a tenth.
constexpr int kNodeTasks = 3000;

template <typename Real, int n>
struct Flow2DShape {
  static constexpr bool F64 = sizeof(Real) == 8;
  static constexpr int Np = n * n, Nb = 4 * (n - 1), LS = n | 1, PS = LS * n, M = n - 2;
  using Val = LineVal<Real>;
  // most threads of a CTA (FP64 and long lines need the registers)
  static constexpr int TMAX = F64 || n > 10 ? 512 : 768;
  static constexpr int COPIES = 4;                       // copies of a node kept in shared memory (more: from L2)
  // learned control: network, V^-1; per element features, hidden layers, transfer function
  static constexpr size_t learned_bytes(int epc) {
    return (size_t)(2 * n * 64 + 64 * 65 + 2 * 64 + 2 * 64 + 2) * sizeof(float) + (size_t)(n * n + 4 * n) * sizeof(Real) + 64 +
           (size_t)epc * ((2 * n + 2 * 64 + 2) * sizeof(Real) + n * sizeof(Val) + n * sizeof(Real) + 2 * sizeof(int));
  }
  // shared memory of one element: f, f^0, sums; weights and rho; wall terms; coefficients; copies
  static constexpr size_t element_bytes(bool affine, bool node) {
    return (node ? (size_t)9 * PS * sizeof(Limb) : 0) +
           (size_t)9 * PS * (2 * sizeof(Real) + sizeof(Val)) + (size_t)(Nb + PS) * sizeof(Real) +
           (size_t)9 * Nb * sizeof(Real) + (affine ? (size_t)18 * sizeof(Val) : (size_t)4 * PS * sizeof(Val)) +
           (size_t)(2 * 9 + 10) * sizeof(int) + (size_t)Nb * (sizeof(Real) + (COPIES + 2) * sizeof(int));
  }
  static constexpr size_t fixed_bytes(bool node) { return (node ? (size_t)n * n * sizeof(Limb) : 0) + (size_t)n * (sizeof(Val) + sizeof(Real)) + (size_t)(Nb + Np + M * M) * sizeof(int) + 64; }
};

// a word of a packet is one 8-byte access on either side, strong and device-wide, so that a reader
// sees its value and its tag together
__device__ __forceinline__ void put_packet(Packet<float> *p, float v, unsigned tag) {
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(&p->w[0]), "l"(((unsigned long long)tag << 32) | __float_as_uint(v))
               : "memory");
}
__device__ __forceinline__ void put_packet(Packet<double> *p, double v, unsigned tag) {
  const unsigned long long t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(&p->w[0]), "l"(t | (unsigned)__double2hiint(v)),
               "l"(t | (unsigned)__double2loint(v))
               : "memory");
}
__device__ __forceinline__ unsigned long long ld_relaxed(const unsigned long long *p) {
  unsigned long long v;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
  return v;
}
// true when the packet carries exchange `tag`
__device__ __forceinline__ bool get_packet(const Packet<float> *p, unsigned tag, float &v) {
  const unsigned long long w = ld_relaxed(&p->w[0]);
  v = __uint_as_float((unsigned)w);
  return (unsigned)(w >> 32) == tag;
}
__device__ __forceinline__ bool get_packet(const Packet<double> *p, unsigned tag, double &v) {
  const unsigned long long h = ld_relaxed(&p->w[0]), l = ld_relaxed(&p->w[1]);
  v = __hiloint2double((int)(unsigned)h, (int)(unsigned)l);
  return (unsigned)(h >> 32) == tag && (unsigned)(l >> 32) == tag;
}

// filter of one line that holds infinities or NaN (FP64 bits at row[k st])
template <int n>
__device__ __noinline__ void slow_filter_row(const FilterMats<double, n> &m, const double *g, long long *row, int st) {
  double d[n];
#pragma unroll 1
  for (int j = 0; j < n; ++j) d[j] = 0;
#pragma unroll 1
  for (int k = 2; k < n; ++k) {
    if (g[k] == 0) continue;
    double s = 0;
#pragma unroll 1
    for (int j = 0; j < n; ++j) s += m.Wd[k][j] * __longlong_as_double(row[j * st]);
#pragma unroll 1
    for (int j = 1; j < n - 1; ++j) d[j] += m.Ud[k][j] * (g[k] * s);
  }
#pragma unroll 1
  for (int j = 1; j < n - 1; ++j) row[j * st] = __double_as_longlong(__longlong_as_double(row[j * st]) + d[j]);
}
// FP64 collision of one node beyond the integers' range (populations at f[a ps])
static __device__ __noinline__ double collide_fp64(double *f, int ps, double rho0, double omega, double dt, double half_dt,
                                                   double gx, double gy, bool forced) {
  double g[9];
  const double acc[3] = {gx, gy, 0.0};
#pragma unroll
  for (int a = 0; a < 9; ++a) g[a] = f[a * ps];
  const double rho = bgk_collide<double, SELBM_D2Q9>(g, rho0, omega, dt, half_dt, acc, forced);
#pragma unroll
  for (int a = 0; a < 9; ++a) f[a * ps] = g[a];
  return rho;
}

__device__ __forceinline__ float as_val(float v) { return v; }
__device__ __forceinline__ long long as_val(double v) { return __double_as_longlong(v); }

// NODE (FP64): one thread per (population, node) and stage instead of lines; see launch_flow2d_t
template <typename Real, int n, bool AFFINE, bool NODE, bool LEARNED>
__global__ void __launch_bounds__(Flow2DShape<Real, n>::TMAX, 1)
flow2d_kernel(const Flow2DArgs<Real> p, const StageMats<Real, n> m, const FilterMats<Real, n> fm, const CollideFix cfix,
              const Learn2DArgs<Real> lc) {
  using S = Flow2DShape<Real, n>;
  using Val = LineVal<Real>;
  constexpr bool F64 = S::F64;
  constexpr int Np = S::Np, Nb = S::Nb, LS = S::LS, PS = S::PS, COPIES = S::COPIES;
  constexpr int SHIFT = FixScale<n>::SHIFT;
  constexpr VelTab V = LT<SELBM_D2Q9>::v;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int epc = p.epc, e0 = blockIdx.x * epc, ne = min(epc, p.E - e0), tid = threadIdx.x, T = blockDim.x;
  Val *X = reinterpret_cast<Val *>(smem_raw);          // [ne][9][PS] sums of the passes
  Val *sge = X + (size_t)epc * 9 * PS;                  // LEARNED: [ne][n] sigma_k - 1 of the elements
  Real *sVi = reinterpret_cast<Real *>(sge + (LEARNED ? (size_t)epc * n : 0));   // LEARNED: [n][n] V^-1, ...
  Real *sX = sVi + (LEARNED ? n * n : 0);               // [ne][2n] features, then scaled inputs
  Real *sH1 = sX + (LEARNED ? epc * 2 * n : 0);         // [ne][64]
  Real *sH2 = sH1 + (LEARNED ? epc * 64 : 0);           // [ne][64]
  Real *sO = sH2 + (LEARNED ? epc * 64 : 0);            // [ne][2]
  Real *slh = sO + (LEARNED ? epc * 2 : 0);             // [4n] lo, hi
  Real *sged = slh + (LEARNED ? 4 * n : 0);             // [ne][n] sigma_k - 1 as a Real
  float *sW1 = reinterpret_cast<float *>(sged + (LEARNED ? epc * n : 0));   // [2n][64] W1 transposed
  float *sW2 = sW1 + (LEARNED ? 2 * n * 64 : 0);        // [64][65] W2 transposed
  float *sb = sW2 + (LEARNED ? 64 * 65 : 0);            // b1[64], b2[64], W3[2][64], b3[2]
  int *sin = reinterpret_cast<int *>(sb + (LEARNED ? 4 * 64 + 2 : 0));      // [ne] features in range
  int *sgs = sin + (LEARNED ? epc : 0);                 // FP64: [ne] shift of sge (filter_gain)
  Val *cf = reinterpret_cast<Val *>(smem_raw + (LEARNED ? (((unsigned char *)(sgs + epc) - smem_raw) + 15) / 16 * 16
                                                        : (size_t)epc * 9 * PS * sizeof(Val)));   // affine [ne][9][2]: -dt e.grad r_l; curved [ne][4][PS]: dr_l/dx_k
  Limb *FQ = reinterpret_cast<Limb *>(cf + (size_t)epc * (AFFINE ? 18 : 4 * PS));   // NODE: [ne][9][PS] f in fixed point
  Limb *sD = FQ + (NODE ? (size_t)epc * 9 * PS : 0);    // NODE: [n][n] D_hat
  Val *sgk = reinterpret_cast<Val *>(sD + (NODE ? n * n : 0));   // [n] sigma_k - 1
  Real *F = reinterpret_cast<Real *>(sgk + n);          // [ne][9][PS] f of the stage
  Real *F0 = F + (size_t)epc * 9 * PS;                  // [ne][9][PS] f^0
  Real *wj = F0 + (size_t)epc * 9 * PS;                 // [ne][Nb] quadrature weights of boundary nodes
  Real *srho = wj + (size_t)epc * Nb;                   // [ne][PS] rho of the step (forcing)
  Real *wb = srho + (size_t)epc * PS;                   // [ne][Nb][9] wall terms (zero off the walls)
  Real *sminv = wb + (size_t)epc * Nb * 9;              // [ne][Nb] 1 / assembled mass
  Real *R = sminv + (size_t)epc * Nb;                   // [9][nrem] fetched shares
  Real *Rb = R + 9 * (size_t)p.rmax;                    // [10][nbas] fetched f^0 and rho of owners
  Real *sgd = Rb + 10 * (size_t)p.bmax;                 // [n]
  int *em = reinterpret_cast<int *>(sgd + n);           // [2][ne][9] tile exponents (FP64), by stage parity
  int *ge = em + 2 * epc * 9;                           // [ne][9] (curved: [ne]) coefficient exponents
  int *sslot = ge + epc * 10;                           // [ne][Nb][COPIES] shares of a boundary node's copies: index of a
                                                        // fetched one, -3 - offset in X of this CTA's, -1 none; first -2: more
  int *sbase = sslot + epc * Nb * COPIES;               // [ne][Nb] where the owner's f^0 is: -1 here, -3 - offset in F0, or fetched
  int *swall = sbase + epc * Nb;                        // [wall points] el Nb + b of this CTA's wall points
  int *srem = swall + epc * Nb;                         // [nrem] trace offsets of the shares to fetch
  int *sbrem = srem + p.rmax;                           // [nbas] shared-node indices of the owners' values to fetch
  int *bi = sbrem + p.bmax;                             // [Nb] tile offset of boundary node b
  int *off = bi + Nb;                                   // [Np] tile offset of local node i
  int *ini = off + Np;                                  // [M M] tile offset of the element-interior nodes
  __shared__ int s_fail, s_flag;
  __shared__ double s_red[2][Flow2DShape<Real, n>::TMAX / 32], s_prev[3];
  __shared__ Real s_t[9], s_c[9];                       // weights; B dt 3 t_a e_a . g / B
  __shared__ signed char s_e[9][2], s_o[9];
  __shared__ Limb s_tc[9];                              // t_a in fixed point

  if (tid < 9) {
    static_for<0, 9>([&](auto ac) {
      constexpr int a = decltype(ac)::value;
      if (a == tid) {
        s_t[a] = Real(V.t[a]);
        s_o[a] = (signed char)V.opp[a];
        s_tc[a] = cfix.t[V.e[a][0] * V.e[a][0] + V.e[a][1] * V.e[a][1]];
        s_e[a][0] = (signed char)V.e[a][0];
        s_e[a][1] = (signed char)V.e[a][1];
        s_c[a] = p.dt * Real(3) * Real(V.t[a]) * (Real(V.e[a][0]) * p.g[0] + Real(V.e[a][1]) * p.g[1]);
      }
    });
  }
  if (tid == 0) s_fail = 0;
  if (tid < n) {
    sgd[tid] = fm.g[tid];
    if constexpr (F64) sgk[tid] = filter_gain(fm.g[tid], filter_gain_shift(fm, fm.ex));
    else sgk[tid] = fm.g[tid];
  }
#pragma unroll 1
  for (int i = tid; i < Np; i += T) {
    const int b = p.bslot[i];
    off[i] = i % n + LS * (i / n);
    if (b >= 0) bi[b] = off[i];
    else ini[(i % n - 1) + S::M * (i / n - 1)] = off[i];
  }
  if constexpr (NODE) {
    // dense D_hat from its even-odd halves (D[n-1-j][n-1-k] = -D[j][k])
    auto val = [](const Limb &l) { return (long long)l.hi * (1ll << 32) + l.lo; };
#pragma unroll 1
    for (int t = tid; t < n * n; t += T) {
      const int j = t / n, k = t - j * n;
      const bool low = 2 * j <= n - 1;
      const int jj = low ? j : n - 1 - j, k2 = low ? k : n - 1 - k;
      const bool left = 2 * k2 <= n - 1;
      const int kk = left ? k2 : n - 1 - k2;
      const long long P = val(m.P[jj][kk]), M = val(m.M[jj][kk]), d = left ? P + M : P - M;
      sD[t] = limbs(low ? d : -d);
    }
  }
#pragma unroll 1
  for (int k = tid; k < 2 * epc * 9; k += T) em[k] = kMinExp;
#pragma unroll 1
  for (int k = tid; k < ne * Nb * 9; k += T) wb[k] = 0;
  __syncthreads();                                       // bi
  const int w0 = p.wall_off[e0], nw = p.wall_off[e0 + ne] - w0;
#pragma unroll 1
  for (int k = tid; k < nw; k += T) {
    int el = 0;
    while (p.wall_off[e0 + el + 1] <= w0 + k) ++el;
    swall[k] = el * Nb + p.walls[w0 + k].b;
  }
  const int r0 = p.rem_off[blockIdx.x], nrem = p.rem_off[blockIdx.x + 1] - r0;
  const int q0 = p.bas_off[blockIdx.x], nbas = p.bas_off[blockIdx.x + 1] - q0;
#pragma unroll 1
  for (int k = tid; k < nrem; k += T) srem[k] = p.rem[r0 + k];
#pragma unroll 1
  for (int k = tid; k < nbas; k += T) sbrem[k] = p.bas[q0 + k];
  // shares and owners inside the CTA: (element, slot) of the tables to offsets in the tiles
  auto local = [&](int s) { return s >= -1 ? s : -3 - ((-3 - s) / Nb * 9 * PS + bi[(-3 - s) % Nb]); };
#pragma unroll 1
  for (int k = tid; k < ne * Nb; k += T) {
    const size_t lg = (size_t)e0 * Nb + k;
    const int c0 = p.loc_off[lg], nc = p.loc_off[lg + 1] - c0;
    sminv[k] = p.minv[p.loc_u[lg]];
    sbase[k] = local(p.loc_base[lg]);
    for (int c = 0; c < COPIES; ++c) sslot[k * COPIES + c] = c < nc ? local(p.loc_slot[c0 + c]) : -1;
    if (nc > COPIES) sslot[k * COPIES] = -2;
  }
  __syncthreads();

  // ---- element constants and the state
#pragma unroll 1
  for (int k = tid; k < ne * Np; k += T) {
    const int el = k / Np, i = k - el * Np, e = e0 + el;
    const int b = p.bslot[i];
    if (b >= 0) wj[el * Nb + b] = AFFINE ? p.el_J[e] * m.w[i % n] * m.w[i / n] : p.wJ[(size_t)e * Np + i];
    if constexpr (!AFFINE) {
      if constexpr (F64) {
        // fixed point at the element's largest exponent
        const int sh = p.gexp[e];
        if (i == 0) ge[el] = sh;
#pragma unroll
        for (int c = 0; c < 4; ++c)
          cf[((size_t)el * 4 + c) * PS + i % n + LS * (i / n)] = __double2ll_rn(scalbn(p.drdx[((size_t)e * Np + i) * 4 + c], sh));
      } else {
#pragma unroll
        for (int c = 0; c < 4; ++c) cf[((size_t)el * 4 + c) * PS + i % n + LS * (i / n)] = p.drdx[((size_t)e * Np + i) * 4 + c];
      }
    }
  }
  if constexpr (AFFINE) {
#pragma unroll 1
    for (int k = tid; k < ne * 9; k += T) {
      const int el = k / 9, a = k - el * 9;
      const Real *g = p.el_drdx + (size_t)(e0 + el) * 4;
      Real c[2];
#pragma unroll
      for (int l = 0; l < 2; ++l) c[l] = -p.dt * (Real(s_e[a][0]) * g[2 * l] + Real(s_e[a][1]) * g[2 * l + 1]);
      if constexpr (F64) {
        const int ex = max(1, max(exp_of(c[0]), exp_of(c[1])));
        ge[k] = 1082 - ex;
#pragma unroll
        for (int l = 0; l < 2; ++l) cf[2 * k + l] = __double2ll_rn(scalbn(c[l], 1082 - ex));
      } else {
        cf[2 * k] = c[0];
        cf[2 * k + 1] = c[1];
      }
    }
  }
  if constexpr (LEARNED) {
    const __nv_bfloat16 *W1 = lc.W, *B1 = W1 + 64 * 2 * n, *W2 = B1 + 64, *B2 = W2 + 64 * 64, *W3 = B2 + 64, *B3 = W3 + 128;
#pragma unroll 1
    for (int k = tid; k < 64 * 2 * n; k += T) sW1[(k % (2 * n)) * 64 + k / (2 * n)] = __bfloat162float(W1[k]);
#pragma unroll 1
    for (int k = tid; k < 64 * 64; k += T) sW2[(k % 64) * 65 + k / 64] = __bfloat162float(W2[k]);
#pragma unroll 1
    for (int k = tid; k < 64; k += T) {
      sb[k] = __bfloat162float(B1[k]);
      sb[64 + k] = __bfloat162float(B2[k]);
      sb[128 + k] = __bfloat162float(W3[k]);
      sb[192 + k] = __bfloat162float(W3[64 + k]);
    }
    if (tid < 2) sb[256 + tid] = __bfloat162float(B3[tid]);
#pragma unroll 1
    for (int k = tid; k < n * n; k += T) sVi[k] = lc.Vinv[k];
    if (tid < 2 * n) { slh[tid] = lc.lo[tid]; slh[2 * n + tid] = lc.hi[tid]; }
    if (tid < 3) s_prev[tid] = lc.acc[2 + tid];
    if (tid == 0) s_flag = *lc.flag;
  }
  auto track = [&](int par, int el, int a, Real v) {     // exponent of a value written to F
    if constexpr (F64) atomicMax(&em[(par * epc + el) * 9 + a], exp_of(v));
  };
  int par = 0;                                           // em[par]: exponents of what F holds
#pragma unroll 1
  for (int k = tid; k < ne * Np; k += T) {
    const int el = k / Np, i = k - el * Np;
    const size_t g = p.l2g[(size_t)(e0 + el) * Np + i];
#pragma unroll
    for (int a = 0; a < 9; ++a) {
      const Real v = p.f[(size_t)a * p.Gs + g];
      F[((size_t)el * 9 + a) * PS + i % n + LS * (i / n)] = v;
      track(par, el, a, v);
    }
  }
  __syncthreads();

  unsigned epoch = p.epoch;
  // the packet of this exchange, polled within a bound
  auto wait_packet = [&](const Packet<Real> *q) -> Real {
    Real v;
    int spin = 0;
    while (!get_packet(q, epoch, v)) {
      if (++spin >= kFlowSpins || ((spin & 4095) == 0 && *(volatile int *)p.abort != 0)) {
        *(volatile int *)p.abort = 1;
        s_fail = 1;
        break;
      }
    }
    return v;
  };
  const bool forced = p.has_force != 0;
  // exponent of a value written to F (FP64), one atomic per population and warp
  auto track_max = [&](int *e9, int q, int e) {
    const unsigned peers = __match_any_sync(__activemask(), q);
    const int top = __reduce_max_sync(peers, e);
    if ((peers & ((1u << (tid & 31)) - 1u)) == 0u) atomicMax(&e9[q], top);
  };
  auto owner_node = [&](int ob) -> int {                 // index in srho of the owner at -3 - ob in F0
    const int at = -3 - ob, el = at / (9 * PS);
    return el * PS + at - el * 9 * PS;
  };
  // body(o, i) for i < CNT of each of `outer` tiles: a warp takes 32 consecutive i of one tile, or
  // several whole tiles where they are short, so that divisions are by warp and not by task
  const int warp = tid >> 5, lane = tid & 31, nwarp = T >> 5;
  auto tiles = [&](auto cntc, int outer, auto body) {
    constexpr int CNT = decltype(cntc)::value;
    if constexpr (CNT > 16) {
      constexpr int CH = (CNT + 31) / 32;
#pragma unroll 1
      for (int w = warp; w < outer * CH; w += nwarp) {
        const int o = w / CH, i = (w - o * CH) * 32 + lane;
        if (i < CNT) body(o, i);
      }
    } else {
      constexpr int PK = 32 / CNT;
      const int sub = lane / CNT, i = lane - sub * CNT;
      if (sub < PK)
#pragma unroll 1
        for (int o = warp * PK + sub; o < outer; o += nwarp * PK) body(o, i);
    }
  };
  using CNp = std::integral_constant<int, Np>;
  using CNb = std::integral_constant<int, Nb>;
  using Cin = std::integral_constant<int, S::M * S::M>;
  using Cn = std::integral_constant<int, n>;
  const int ntile = 9 * ne;

  // packets of other CTAs into shared memory: a thread looks at two before it waits for one
        auto fetch = [&](int pops, int count, auto address, Real *dst) {   // dst [pops][count]
          constexpr int U = 2;
          const int blocks = (count + 31) >> 5;
  #pragma unroll 1
          for (int w = warp; w < pops * blocks; w += U * nwarp) {
            Real v[U];
            const Packet<Real> *src[U];
            Real *to[U];
            bool ok[U];
  #pragma unroll
            for (int c = 0; c < U; ++c) {
              const int wc = w + c * nwarp, a = wc / blocks, r = (wc - a * blocks) * 32 + lane;
              ok[c] = true;
              to[c] = nullptr;
              if (wc < pops * blocks && r < count) {
                src[c] = address(a, r);
                to[c] = dst + a * count + r;
                ok[c] = get_packet(src[c], epoch, v[c]);
              }
            }
  #pragma unroll
            for (int c = 0; c < U; ++c) {
              if (!ok[c]) v[c] = wait_packet(src[c]);
              if (to[c]) *to[c] = v[c];
            }
          }
        };
  // sum of the shares of local boundary node b's copies, population tile q, in ascending copy order
  auto copies_sum = [&](int q, int b) -> Real {
    const int el = q / 9, a = q - 9 * el, lb = el * Nb + b;
    const Real *xa = reinterpret_cast<const Real *>(X) + a * PS, *ra = R + a * nrem;
    const int *sl = sslot + lb * COPIES;
    Real sum = 0;
    if (sl[0] != -2) {
#pragma unroll
      for (int c = 0; c < COPIES; ++c) {
        const int s = sl[c];
        if (s != -1) sum += s >= 0 ? ra[s] : xa[-3 - s];
      }
    } else {
      const size_t lg = (size_t)e0 * Nb + lb;
#pragma unroll 1
      for (int c = p.loc_off[lg]; c < p.loc_off[lg + 1]; ++c) {
        const int s = local(p.loc_slot[c]);
        sum += s >= 0 ? ra[s] : xa[-3 - s];
      }
    }
    return sum;
  };

  // The phases are rolled loops over axes, populations and nodes where that costs little: the code
  // of a step has to stay in the instruction cache, since every phase runs it once.
#pragma unroll 1
  for (int step = 0; step < p.nsteps; ++step) {
    const bool filt = p.filter && (step > 0 || p.pending);
    const bool owners = filt && !LEARNED;                  // copies filtered apart: the owner's f^0 stands
    const int pass = LEARNED ? lc.pass + step - (p.pending ? 0 : 1) : 0;   // control pass of this step
    const unsigned pass_tag = epoch + 1;
    // ---- learned control: the element's transfer function from the modal energies of rho - rho0
    //      and |u|, the drift sums, the network (BF16 weights)
    if (LEARNED && filt) {
      Real *fld = reinterpret_cast<Real *>(X);             // [ne][9][PS]: planes 0, 1 of each element
      double pm = 0, pk = 0;
      tiles(CNp{}, ne, [&](int el, int i) {
        const int o = off[i], at = el * 9 * PS + o;
        Real drho = 0, jx = 0, jy = 0;
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          const Real v = F[at + a * PS];
          drho += v;
          if (V.e[a][0] > 0) jx += v;
          else if (V.e[a][0] < 0) jx -= v;
          if (V.e[a][1] > 0) jy += v;
          else if (V.e[a][1] < 0) jy -= v;
        }
        const Real rho = p.rho0 + drho, ux = jx / rho, uy = jy / rho, uu = ux * ux + uy * uy;
        fld[at] = drho;
        fld[at + PS] = sqrt(uu);
        const Real wq = AFFINE ? p.el_J[e0 + el] * m.w[i % n] * m.w[i / n] : p.wJ[(size_t)(e0 + el) * Np + i];
        pm += wide(wq) * wide(rho);
        pk += wide(wq) * wide(uu);
      });
      pm = warp_sum(pm);
      pk = warp_sum(pk);
      if (lane == 0) { s_red[0][warp] = pm; s_red[1][warp] = pk; }
      __syncthreads();
      if (tid < 2) {
        double s = 0;
        for (int w = 0; w < nwarp; ++w) s += s_red[tid][w];
        if (tid == 1) s *= 0.5 * (double)p.rho0;
        put_packet(lc.sums + ((size_t)(pass & 1) * gridDim.x + blockIdx.x) * 2 + tid, s, epoch + 1);
      }
#pragma unroll 1
      for (int ax = 0; ax < 2; ++ax) {
        const int lst = ax ? 1 : LS, stp = ax ? LS : 1;
        tiles(Cn{}, 2 * ne, [&](int q, int L) {
          Real *row = fld + ((q >> 1) * 9 + (q & 1)) * PS + lst * L;
          Real v[n];
#pragma unroll
          for (int k = 0; k < n; ++k) v[k] = row[k * stp];
#pragma unroll 1
          for (int j = 0; j < n; ++j) {
            Real s = 0;
#pragma unroll
            for (int k = 0; k < n; ++k) s += sVi[j * n + k] * v[k];
            row[j * stp] = s;
          }
        });
        if (tid < ne) sin[tid] = 1;
        __syncthreads();
      }
      // shell k: modes whose larger index is k
      tiles(Cn{}, 2 * ne, [&](int q, int k) {
        const int el = q >> 1, fi = q & 1;
        const Real *c = fld + (el * 9 + fi) * PS;
        Real s = 0;
        for (int i = 0; i <= k; ++i) s += c[i + LS * k] * c[i + LS * k];
        for (int i = 0; i < k; ++i) s += c[k + LS * i] * c[k + LS * i];
        const Real x = log10(s + Real(1e-30)), lo = slh[fi * n + k], hi = slh[2 * n + fi * n + k];
        if (!(x >= lo && x <= hi)) sin[el] = 0;
        sX[el * 2 * n + fi * n + k] = Real(2) * (x - lo) / (hi - lo) - Real(1);
      });
      __syncthreads();
      using C64 = std::integral_constant<int, 64>;
      tiles(C64{}, ne, [&](int el, int o) {
        Real z = (Real)sb[o];
        for (int i = 0; i < 2 * n; ++i) z += (Real)sW1[i * 64 + o] * sX[el * 2 * n + i];
        sH1[el * 64 + o] = tanh(z);
      });
      __syncthreads();
      tiles(C64{}, ne, [&](int el, int o) {
        Real z = (Real)sb[64 + o];
        for (int i = 0; i < 64; ++i) z += (Real)sW2[i * 65 + o] * sH1[el * 64 + i];
        sH2[el * 64 + o] = tanh(z);
      });
      __syncthreads();
#pragma unroll 1
      for (int t = warp; t < 2 * ne; t += nwarp) {
        const int el = t >> 1, o = t & 1;
        Real z = (Real)sb[128 + 64 * o + lane] * sH2[el * 64 + lane] + (Real)sb[128 + 64 * o + 32 + lane] * sH2[el * 64 + 32 + lane];
        z = warp_sum(z);
        if (lane == 0) sO[t] = z + (Real)sb[256 + o];
      }
      __syncthreads();
      tiles(Cn{}, ne, [&](int el, int k) {
        const bool use_net = sin[el] && !s_flag;
        Real g = fm.g[k], last = 0;                         // last: g of the highest mode, the largest
        if (use_net) {
          const Real gam = Real(0.5) / (Real(1) + exp(-sO[2 * el])), kc = Real(2) + Real(n - 4) / (Real(1) + exp(-sO[2 * el + 1]));
          g = 0;
          last = (Real(1) - gam) - Real(1);
          if (k > kc) {
            const Real r = (Real(k) - kc) / (Real(n - 1) - kc);
            // sigma = 1 - gamma r^2 rounded as the transfer function that is handed out
            g = (Real(1) - gam * r * r) - Real(1);
          }
        } else if (k == 0) {
          atomicAdd(lc.n_fallback, 1);
        }
        sged[el * n + k] = g;
        if constexpr (F64) {
          const int sh = filter_gain_shift(fm, use_net ? exp_of(last) : fm.ex);
          sge[el * n + k] = filter_gain(g, sh);
          if (k == 0) sgs[el] = sh;
        } else sge[el * n + k] = g;
        lc.sigma_out[(size_t)(e0 + el) * n + k] = g + Real(1);
      });
      __syncthreads();
    }
    // ---- explicit filter of the previous step (Sec. 2.4), r- then s-lines
    if (filt) {
      Val *Y = X;                                           // FP64: the tile in fixed point
      if constexpr (F64) {
        tiles(CNp{}, ntile, [&](int q, int i) {
          const int ex = em[par * epc * 9 + q], at = q * PS + off[i];
          X[at] = ex == 2047 ? __double_as_longlong(F[at]) : to_fixed<kFilterShift>(F[at], ex);
        });
        __syncthreads();
      } else Y = F;
#pragma unroll 1
      for (int ax = 0; ax < 2; ++ax) {
        const int lst = ax ? 1 : LS, st = ax ? LS : 1;
        tiles(Cn{}, ntile, [&](int q, int L) {
          Val *row = Y + q * PS + lst * L;
          Val v[n];
#pragma unroll
          for (int k = 0; k < n; ++k) v[k] = row[k * st];
          if constexpr (F64) {
            if (em[par * epc * 9 + q] == 2047) {
              slow_filter_row<n>(fm, LEARNED ? sged + q / 9 * n : sgd, row, st);
              return;
            }
            if constexpr (LEARNED) line_filter<n>(fm, sge + q / 9 * n, sgs[q / 9], v);
            else line_filter<n>(fm, sgk, filter_gain_shift(fm, fm.ex), v);
          } else line_filter<n>(fm, LEARNED ? sge + q / 9 * n : sgk, v);
#pragma unroll
          for (int k = 1; k < n - 1; ++k) row[k * st] = v[k];
        });
        __syncthreads();
      }
      if constexpr (F64) {
        tiles(CNp{}, ntile, [&](int q, int i) {
          const int ex = em[par * epc * 9 + q], at = q * PS + off[i];
          // the tile's change alone, see lines_filter_kernel
          F[at] = ex == 2047 ? __longlong_as_double(X[at])
                             : F[at] + from_fixed(X[at] - to_fixed<kFilterShift>(F[at], ex), ex - (1023 + 52 + kFilterShift));
        });
        __syncthreads();
      }
    }
    // ---- element-dependent filters: the copies of a shared node take their mass-weighted average
    if (LEARNED && filt) {
      ++epoch;
      Packet<Real> *Tb = reinterpret_cast<Packet<Real> *>(p.T) + (size_t)(epoch & 1u) * p.E * Nb * 9;
      tiles(CNb{}, ntile, [&](int q, int b) {
        const int at = q * PS + bi[b];
        const Real v = wj[q / 9 * Nb + b] * F[at];
        put_packet(Tb + (e0 * 9 + q) * Nb + b, v, epoch);
        X[at] = as_val(v);
      });
      fetch(9, nrem, [&](int a, int r) { return Tb + srem[r] + a * Nb; }, R);
      __syncthreads();
      tiles(CNb{}, ntile, [&](int q, int b) { F[q * PS + bi[b]] = copies_sum(q, b) * sminv[q / 9 * Nb + b]; });
      __syncthreads();
      if (s_fail) return;
    }
    // ---- BGK collision at every local node; after a filter the owner's f^0 of a shared node
    //      stands for all copies (their lines were filtered in different element frames)
    auto publish = [&](int el, int i, int a, Real v) {
      const int b = p.bslot[i];
      if (b >= 0 && p.owner[(size_t)(e0 + el) * Np + i])
        put_packet(reinterpret_cast<Packet<Real> *>(p.base) + (size_t)p.loc_u[(size_t)(e0 + el) * Nb + b] * 10 + a, v, epoch + 1);
    };
    if constexpr (F64) {
      // per node the moments and products (see collide_fixed), kept in X: base, P_xx, P_yy, S_xy,
      // j_x, j_y, exponent (0: the node took the FP64 collision), X of the rest population
      int *emn = em + (par ^ 1) * epc * 9;
#pragma unroll 1
      for (int k = tid; k < epc * 9; k += T) emn[k] = kMinExp;
      tiles(CNp{}, ne, [&](int el, int i) {
        const int at = el * 9 * PS + off[i];
        int ex = kMinExp;
#pragma unroll 3
        for (int a = 0; a < 9; ++a) ex = max(ex, exp_of(F[at + a * PS]));
        long long sr = 0, sx = 0, sy = 0;
#pragma unroll 3
        for (int a = 0; a < 9; ++a) {
          const long long v = to_fixed_rn<kColShift>(F[at + a * PS], ex);
          sr += v;
          sx += s_e[a][0] * v;
          sy += s_e[a][1] * v;
        }
        const int sc = ex - (1023 + 52 + kColShift);
        double rho = p.rho0 + from_fixed(sr, sc);
        const double inv = 1.0 / rho;
        double vx = from_fixed(sx, sc) * inv, vy = from_fixed(sy, sc) * inv;
        if (forced) { vx += cfix.kappa2 * p.g[0]; vy += cfix.kappa2 * p.g[1]; }
        const long long js = ((sx < 0 ? -sx : sx) >> 1) + ((sy < 0 ? -sy : sy) >> 1);
        if (!fix_in_range<2>(ex, max(exp_of(vx), exp_of(vy)), 2 * js)) ex = 0;
        X[at + 6 * PS] = ex;
        if (ex == 0) {
          rho = collide_fp64(F + at, PS, p.rho0, p.omega, p.dt, p.half_dt, p.g[0], p.g[1], forced);
        } else {
          const Limb jx = limbs(sx), jy = limbs(sy), ux = limbs(fix_velocity(vx)), uy = limbs(fix_velocity(vy));
          Fix128 xx{0, 0}, yy{0, 0}, xy{0, 0};
          fix_mac(xx, jx, ux);
          fix_mac(yy, jy, uy);
          fix_mac(xy, jx, uy);
          fix_mac(xy, jy, ux);
          const long long P = fix_product(xx), R = fix_product(yy);
          X[at] = fix_base4(sr, P + R);
          X[at + PS] = P;
          X[at + 2 * PS] = R;
          X[at + 3 * PS] = fix_product(xy);
          X[at + 4 * PS] = sx;
          X[at + 5 * PS] = sy;
          X[at + 7 * PS] = fix_rest(sr, P + R);
        }
        if (forced) {
          srho[el * PS + off[i]] = rho;
          if (owners) publish(el, i, 9, rho);
        }
      });
      __syncthreads();
      tiles(CNp{}, ntile, [&](int q, int i) {
        const int el = q / 9, a = q - 9 * el, o = off[i], at = q * PS + o;
        const Val *x = X + el * 9 * PS + o;
        const int ex = (int)x[6 * PS];
        double v = F[at];
        if (ex != 0) {
          const int cx = s_e[a][0], cy = s_e[a][1];
          const long long even = (cx ? x[PS] : 0) + (cy ? x[2 * PS] : 0) + cx * cy * x[3 * PS];
          const long long x4 = x[0] + fix_even4(even) + 3 * fix_quarter(cx * x[4 * PS] + cy * x[5 * PS]);
          v += fix_change(cfix, s_tc[a], a == 0 ? x[7 * PS] : x4, to_fixed_rn<kColShift>(v, ex), ex);
        }
        F[at] = v;
        F0[at] = v;
        if (owners) publish(el, i, a, v);
        track_max(emn, q, exp_of(v));
      });
    } else {
      tiles(CNp{}, ne, [&](int el, int i) {
        const int at = el * 9 * PS + off[i];
        Real f[9];
#pragma unroll
        for (int a = 0; a < 9; ++a) f[a] = F[at + a * PS];
        const Real rho = bgk_collide<Real, SELBM_D2Q9>(f, p.rho0, p.omega, p.dt, p.half_dt, p.g, forced);
#pragma unroll
        for (int a = 0; a < 9; ++a) {
          F[at + a * PS] = f[a];
          F0[at + a * PS] = f[a];
        }
        if (forced) srho[el * PS + off[i]] = rho;
        if (owners) {
          const int b = p.bslot[i];
          if (b >= 0 && p.owner[(size_t)(e0 + el) * Np + i]) {
            Packet<Real> *base = reinterpret_cast<Packet<Real> *>(p.base) + (size_t)p.loc_u[(size_t)(e0 + el) * Nb + b] * 10;
#pragma unroll
            for (int a = 0; a < 9; ++a) put_packet(base + a, f[a], epoch + 1);
            if (forced) put_packet(base + 9, rho, epoch + 1);
          }
        }
      });
    }
    par ^= 1;
    __syncthreads();

    // ---- three Runge-Kutta stages
#pragma unroll 1
    for (int st = 0; st < 3; ++st) {
      ++epoch;
      const Real B = st == 0 ? Real(1) : (st == 1 ? Real(0.25) : Real(2.0 / 3.0));
      const int *emc = em + par * epc * 9;
      int *emn = em + (par ^ 1) * epc * 9;
      auto coef = [&](int ax, int q, int a, int off) -> Val {     // coefficient of an axis at a node
        if constexpr (AFFINE) return cf[2 * q + ax];
        else {
          const Val *g = cf + ((size_t)(q / 9) * 4 + 2 * ax) * PS + off;
          return (Val)s_e[a][0] * g[0] + (Val)s_e[a][1] * g[PS];
        }
      };
      if (F64)
#pragma unroll 1
        for (int k = tid; k < epc * 9; k += T) emn[k] = kMinExp;
      // flux bounce-back terms (Sec. 2.2.1), times B when the shares are written
#pragma unroll 1
      for (int idx = tid; idx < 9 * nw; idx += T) {
        const int k = idx / 9, a = idx - 9 * k, lb = swall[k], el = lb / Nb;
        const WallPt<Real> &wp = p.walls[w0 + k];
        const Real *fw = F + (size_t)el * 9 * PS + bi[lb - el * Nb];
        const Real diff = fw[a * PS] - fw[s_o[a] * PS], t6 = Real(6) * s_t[a] * p.rho0;
        const int cx = s_e[a][0], cy = s_e[a][1];
        auto dot = [&](Real x, Real y) -> Real { return (cx > 0 ? x : (cx < 0 ? -x : Real(0))) + (cy > 0 ? y : (cy < 0 ? -y : Real(0))); };
        Real sum = 0;
#pragma unroll 1
        for (int f = 0; f < wp.nf; ++f) {
          const Real *ub = p.wall_u + 3 * (wp.wid[f] - 1);
          const Real nu = dot(wp.n[f][0], wp.n[f][1]);
          if (nu < Real(0)) sum += wp.wsJs[f] * nu * (diff - t6 * dot(ub[0], ub[1]));
        }
        wb[lb * 9 + a] = p.dt * sum;
      }
      // a tile with infinities or NaN: the node's sum in FP64, kept as FP64 bits in X
      auto slow_sum = [&](int q, int i) {
        if constexpr (F64) {
          const int a = q % 9, i0 = i % n, i1 = i / n, o = i0 + LS * i1, sh = ge[AFFINE ? q : q / 9];
          const Real *fr = F + (size_t)q * PS + LS * i1, *fs = F + (size_t)q * PS + i0;
          const double c0 = from_fixed(coef(0, q, a, o), -sh), c1 = from_fixed(coef(1, q, a, o), -sh);
          double sr = 0, ss = 0;
#pragma unroll 1
          for (int k = 0; k < n; ++k) {
            if (c0 != 0) sr += m.D[i0 * n + k] * fr[k];
            if (c1 != 0) ss += m.D[i1 * n + k] * fs[LS * k];
          }
          X[(size_t)q * PS + o] = __double_as_longlong(c0 * sr + c1 * ss);
        }
      };
      if constexpr (NODE) {
        tiles(CNp{}, ntile, [&](int q, int i) {
          const int at = q * PS + off[i];
          if (emc[q] == 2047) slow_sum(q, i);
          else FQ[at] = limbs(to_fixed<SHIFT>(F[at], emc[q]));
        });
      } else {
        // sums of c_l (D_l f) over r-, then s-lines
#pragma unroll 1
        for (int ax = 0; ax < 2; ++ax) {
          const int lst = ax ? 1 : LS, stp = ax ? LS : 1;
          tiles(Cn{}, ntile, [&](int q, int L) {
            const int a = q % 9;
            const Real *row = F + q * PS + lst * L;
            Val *dst = X + q * PS + lst * L;
            Val v[n], d[n];
            const int ex = F64 ? emc[q] : 0;
            if (a == 0) return;
            if (F64 && ex == 2047) {
              if (ax == 0)
                for (int j = 0; j < n; ++j) slow_sum(q, L * n + j);
              return;
            }
#pragma unroll
            for (int k = 0; k < n; ++k) {
              if constexpr (F64) v[k] = to_fixed<SHIFT>(row[k * stp], ex);
              else v[k] = row[k * stp];
            }
            line_deriv<n>(m, v, d);
#pragma unroll
            for (int j = 0; j < n; ++j) {
              const Val c = coef(ax, q, a, lst * L + j * stp);
              const Val old = ax ? dst[j * stp] : Val(0);
              if constexpr (F64) {
                Fix128 y{0, 0};
                fix_mac(y, limbs(c), limbs(d[j]));
                dst[j * stp] = old + fix_top<0>(y);
              } else dst[j * stp] = old + c * d[j];
            }
          });
          if (ax == 0) __syncthreads();
        }
      }
      __syncthreads();
      // boundary nodes publish their weighted share first: it travels while the interior nodes
      // take their stage value
      Packet<Real> *Tb = reinterpret_cast<Packet<Real> *>(p.T) + (size_t)(epoch & 1u) * p.E * Nb * 9;
      const Real sc = AFFINE ? B : -p.dt * B;             // curved coefficients carry no -dt
      auto sum_at = [&](int q, int a, int o) -> Real {     // finished sum of a node
        const int at = q * PS + o;
        if (a == 0) return Real(0);
        if constexpr (F64) {
          const int ex = emc[q], sh = ge[AFFINE ? q : q / 9], xx = 125 - sh - m.cb + ex - FixScale<n>::EXP0;
          if (ex == 2047) return __longlong_as_double(X[at]);
          if constexpr (NODE) {
            const int i1 = o / LS, i0 = o - LS * i1;
            const Limb *fr = FQ + q * PS + LS * i1, *fs = FQ + q * PS + i0;
            const Limb *dr = sD + n * i0, *ds = sD + n * i1;
            Fix128 sr{0, 0}, ss{0, 0}, y{0, 0};
#pragma unroll 3
            for (int c = 0; c < n; ++c) {
              fix_mac_line<n>(sr, dr[c], fr[c]);
              fix_mac_line<n>(ss, ds[c], fs[LS * c]);
            }
            fix_mac(y, limbs(coef(0, q, a, o)), limbs(fix_top<3>(sr)));
            fix_mac(y, limbs(coef(1, q, a, o)), limbs(fix_top<3>(ss)));
            return from_fixed(fix_top<0>(y), xx);
          } else return from_fixed(X[at], xx);
        } else return X[at];
      };
      tiles(CNb{}, ntile, [&](int q, int b) {
        const int el = q / 9, a = q - 9 * el, o = bi[b];
        Real v = wj[el * Nb + b] * (sc * sum_at(q, a, o));
        if (nw > 0) v += B * wb[(el * Nb + b) * 9 + a];
        put_packet(Tb + (e0 * 9 + q) * Nb + b, v, epoch);
        X[q * PS + o] = as_val(v);
      });
      tiles(Cin{}, ntile, [&](int q, int i) {
        const int el = q / 9, a = q - 9 * el, o = ini[i], at = q * PS + o;
        // A f^0 + B (f^{s-1} + x) as f^0 + B (f^{s-1} - f^0 + x), A = 1 - B: one rounding at the
        // size of f (in FP32 the products A f^0 and B f rounded apart drift by 1e-7 of f a step)
        const Real f0v = F0[at];
        Real x = AFFINE ? sum_at(q, a, o) : -p.dt * sum_at(q, a, o);
        if (forced) x += s_c[a] * srho[el * PS + o];
        const Real v = f0v + B * (F[at] - f0v + x);
        F[at] = v;
        if (F64) track_max(emn, q, exp_of(v));
      });
      // the shares of other CTAs (and after a filter the owners' f^0)
      const bool owner_base = st == 0 && owners;
      fetch(9, nrem, [&](int a, int r) { return Tb + srem[r] + a * Nb; }, R);
      if (owner_base)
        fetch(forced ? 10 : 9, nbas,
              [&](int a, int r) { return reinterpret_cast<const Packet<Real> *>(p.base) + (size_t)sbrem[r] * 10 + a; }, Rb);
      __syncthreads();
      // assembly at the element-boundary nodes: f^0 + B (f^{s-1} - f^0) + sum_c T_c / M + B dt F*
      tiles(CNb{}, ntile, [&](int q, int b) {
        const int el = q / 9, a = q - 9 * el, lb = el * Nb + b, o = bi[b], at = q * PS + o;
        const Real sum = copies_sum(q, b);
        Real f0v = F0[at], fv = F[at];
        const int ob = owner_base ? sbase[lb] : -1;
        if (ob != -1) f0v = fv = ob >= 0 ? Rb[a * nbas + ob] : F0[-3 - ob + a * PS];
        Real y = sum * sminv[lb] + B * (fv - f0v);
        if (forced) {
          Real r = srho[el * PS + o];
          if (ob >= 0) r = Rb[9 * nbas + ob];
          else if (ob != -1) r = srho[owner_node(ob)];
          y += B * s_c[a] * r;
        }
        y += f0v;
        F[at] = y;
        if (F64) track_max(emn, q, exp_of(y));
      });
      // learned control, last stage: the drift sums of this step's pass over all CTAs, in a fixed
      // order, against those of the pass before (the fallback holds from the next pass on)
      if (LEARNED && st == 2 && filt && warp == nwarp - 1) {
        double sum[2] = {0, 0};
#pragma unroll 1
        for (int c = lane; c < (int)gridDim.x; c += 32)
#pragma unroll 1
          for (int k = 0; k < 2; ++k) {
            const Packet<double> *src = lc.sums + ((size_t)(pass & 1) * gridDim.x + c) * 2 + k;
            double v;
            int spin = 0;
            while (!get_packet(src, pass_tag, v)) {
              if (++spin >= kFlowSpins || ((spin & 4095) == 0 && *(volatile int *)p.abort != 0)) {
                *(volatile int *)p.abort = 1;
                s_fail = 1;
                break;
              }
            }
            sum[k] += v;
          }
        sum[0] = warp_sum(sum[0]);
        sum[1] = warp_sum(sum[1]);
        if (lane == 0) {
          if (s_prev[2] != 0.0) {
            const double dm = fabs(sum[0] - s_prev[0]) / fabs(s_prev[0]);
            const bool up = lc.check_ke && lc.ke_bound > 0.0 && sum[1] > s_prev[1] * (1.0 + lc.ke_bound);
            if (dm > lc.mass_bound || up) s_flag = 1;
          }
          s_prev[0] = sum[0];
          s_prev[1] = sum[1];
          s_prev[2] = 1.0;
        }
      }
      __syncthreads();
      if (s_fail) return;
      // the owner's f^0 and rho stand for all copies in the later stages too (the owners' own
      // entries are not written)
      if (owner_base) {
        tiles(CNb{}, ntile, [&](int q, int b) {
          const int el = q / 9, a = q - 9 * el, ob = sbase[el * Nb + b];
          if (ob == -1) return;
          F0[q * PS + bi[b]] = ob >= 0 ? Rb[a * nbas + ob] : F0[-3 - ob + a * PS];
          if (forced && a == 0) srho[el * PS + bi[b]] = ob >= 0 ? Rb[9 * nbas + ob] : srho[owner_node(ob)];
        });
        __syncthreads();
      }
      par ^= 1;
    }
  }
  if (LEARNED && blockIdx.x == 0) {
    if (tid < 3) lc.acc[2 + tid] = s_prev[tid];
    if (tid == 0) *lc.flag = s_flag;
  }
  // ---- the state back to the unique nodes (every copy of a shared node holds the same bits)
#pragma unroll 1
  for (int k = tid; k < ne * Np; k += T) {
    const int el = k / Np, i = k - el * Np;
    if (!p.owner[(size_t)(e0 + el) * Np + i]) continue;
    const size_t g = p.l2g[(size_t)(e0 + el) * Np + i];
#pragma unroll
    for (int a = 0; a < 9; ++a) p.f[(size_t)a * p.Gs + g] = F[((size_t)el * 9 + a) * PS + i % n + LS * (i / n)];
  }
}

// L2D: the kernels with the learned control
template <typename Real, int n, bool L2D>
cudaError_t launch_flow2d_t(const Flow2DArgs<Real> &p, const SplitHost &h, bool affine, bool probe,
                            const Learn2DArgs<Real> *lc, bool *fits, cudaStream_t s) {
  using S = Flow2DShape<Real, n>;
  int dev = 0, sms = 0, most = 0, coop = 0;
  cudaError_t e;
  if ((e = cudaGetDevice(&dev)) || (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) ||
      (e = cudaDeviceGetAttribute(&most, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev)) ||
      (e = cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev)))
    return e;
  const size_t fetched = p.rmax * (9 * sizeof(Real) + sizeof(int)) + p.bmax * (10 * sizeof(Real) + sizeof(int));
  auto bytes = [&](bool node) {
    return S::fixed_bytes(node) + p.epc * S::element_bytes(affine, node) + fetched + (lc ? S::learned_bytes(p.epc) : 0);
  };
  const int grid = (p.E + p.epc - 1) / p.epc;
  if (probe) {
    *fits = coop && bytes(false) <= (size_t)most - 1024;
    if (!*fits) return cudaSuccess;
  }
  auto go = [&](auto ac, auto nc, auto lrn) -> cudaError_t {
    constexpr bool AFFINE = decltype(ac)::value, NODE = decltype(nc)::value, LEARNED = decltype(lrn)::value;
    const size_t smem = bytes(NODE);
    // a warp per tile of the boundary passes, more where a thread takes a node
    const int T = std::min(S::TMAX, 32 * std::max(4, 9 * p.epc * (NODE ? (S::Np + 31) / 32 : 1)));
    cudaError_t err = raise_smem<flow2d_kernel<Real, n, AFFINE, NODE, LEARNED>>(smem);
    if (err != cudaSuccess) return err;
    if (probe) {
      int ctas = 0;
      err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&ctas, flow2d_kernel<Real, n, AFFINE, NODE, LEARNED>, T, smem);
      *fits = err == cudaSuccess && grid <= ctas * sms;
      return err;
    }
    StageMats<Real, n> m = make_stage_mats<Real, n>(h);
    FilterMats<Real, n> fm = make_filter_mats<Real, n>(h);
    Flow2DArgs<Real> a = p;
    CollideFix cf = make_collide_fix<SELBM_D2Q9>((double)p.omega, (double)p.dt);
    Learn2DArgs<Real> la = lc ? *lc : Learn2DArgs<Real>{};
    void *args[] = {&a, &m, &fm, &cf, &la};
    return cudaLaunchCooperativeKernel((const void *)flow2d_kernel<Real, n, AFFINE, NODE, LEARNED>, dim3(grid),
                                       dim3(T), args, smem, s);
  };
  using Yes = std::true_type;
  using No = std::false_type;
  if constexpr (L2D) {
    return affine ? go(Yes{}, No{}, Yes{}) : go(No{}, No{}, Yes{});
  } else {
    if constexpr (S::F64) {
      if (p.epc * 9 * S::Np <= kNodeTasks && bytes(true) <= (size_t)most - 1024)
        return affine ? go(Yes{}, Yes{}, No{}) : go(No{}, Yes{}, No{});
    }
    return affine ? go(Yes{}, No{}, No{}) : go(No{}, No{}, No{});
  }
}

// translation units: part 0 without the learned control (FP64: N <= 8), 1 FP64 above, 2 with it
template <typename Real, int PART>
cudaError_t flow2d_part(int N, bool affine, bool probe, const Flow2DArgs<Real> &p, const SplitHost &h, const Learn2DArgs<Real> *lc,
                        bool *fits, cudaStream_t s);

}  // namespace slb
