// State import and read-back: initial state, fields on unique nodes and at local nodes, the
// state at local nodes, diagnostic sums.
//
// These run between steps, once per checkpoint, and were FP64-bound (two FP64 operations a clock
// and SM): about 100 FP64 operations per local node for the moments, 400 for the initial state.
// Moments are now summed in fixed point (selbm_moments.cuh) once per unique node and copied to
// the local nodes; the equilibrium is evaluated per pair of opposite velocities, whose even and
// odd parts are shared.  Taylor-Green 16^3, N = 7, D3Q27, FP32 state.
#include <cuda_runtime.h>

#include <algorithm>

#include "selbm_kernels.cuh"
#include "selbm_moments.cuh"

namespace slb {

static int blocks_for(size_t n) { return (int)std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 152 * 16)); }

// f_bar = f^eq(rho, u) - dt/2 F** stored as g = f_bar - t rho0 (Sec. 2.1, f at equilibrium)
template <typename Real, int LAT>
__global__ void __launch_bounds__(256) init_kernel(const double *rho, const double *u, const int32_t *first, int G, int Gs,
                                                   double rho0, double half_dt, double gx, double gy, double gz,
                                                   int has_force, const Real *fS, double amp, Real *out) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, DIM = V.D;
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    const size_t q = first[g];
    const double r = rho[q];
    double uv[3] = {0, 0, 0}, F[3] = {0, 0, 0}, gg[3] = {gx, gy, gz}, uu = 0, uF = 0;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      uv[k] = u[q * DIM + k];
      uu += uv[k] * uv[k];
    }
    if (has_force) {
#pragma unroll
      for (int k = 0; k < DIM; ++k) {
        if (fS) gg[k] += amp * (double)fS[(size_t)k * G + g];
        F[k] = r * gg[k];
        uF += uv[k] * F[k];
      }
    }
    const double drho = r - rho0, ruu = 1.5 * r * uu;
    static_for<0, Q>([&](auto ac) {
      constexpr int a = decltype(ac)::value, o = V.opp[a];
      if constexpr (o >= a) {
        double eu = 0, eF = 0;
#pragma unroll
        for (int k = 0; k < DIM; ++k) {
          if (V.e[a][k] > 0) { eu += uv[k]; eF += F[k]; }
          else if (V.e[a][k] < 0) { eu -= uv[k]; eF -= F[k]; }
        }
        const double t = V.t[a];
        // even and odd parts of the equilibrium; F** is even
        double even = t * (drho - ruu);
        if constexpr (o != a) even += (4.5 * t * r * eu) * eu;
        if (has_force) even -= half_dt * (t * (9.0 * eu * eF - 3.0 * uF));
        const double odd = 3.0 * t * r * eu;
        out[(size_t)a * Gs + g] = (Real)(even + odd);
        if constexpr (o != a) out[(size_t)o * Gs + g] = (Real)(even - odd);
      }
    });
  }
}

// rho and u on unique nodes, fld [1 + dim][G]; DIAG: per-block partial sums of mass, momentum[3],
// kinetic energy and the non-finite count (summed in block order afterwards)
template <typename Real, int LAT, bool DIAG>
__global__ void __launch_bounds__(256) node_fields_kernel(const Real *buf, int G, int Gs, double rho0, double *fld,
                                                          const double *mass, double *partial) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, DIM = V.D;
  double acc[6] = {0, 0, 0, 0, 0, 0};
  for (int g = blockIdx.x * blockDim.x + threadIdx.x; g < G; g += gridDim.x * blockDim.x) {
    Real f[Q];
#pragma unroll
    for (int a = 0; a < Q; ++a) f[a] = buf[(size_t)a * Gs + g];
    double drho, j[3];
    const int bad = node_moments<LAT>(f, drho, j);
    const double r = rho0 + drho, inv = 1.0 / r;
    double uu = 0;
    if (fld) fld[g] = r;
#pragma unroll
    for (int k = 0; k < DIM; ++k) {
      const double uk = j[k] * inv;
      if (fld) fld[(size_t)(1 + k) * G + g] = uk;
      if (DIAG) uu += uk * uk;
    }
    if (DIAG) {
      const double M = mass[g];
      acc[0] += M * r;
#pragma unroll
      for (int k = 0; k < DIM; ++k) acc[1 + k] += M * j[k];
      acc[4] += M * uu;
      if (bad) acc[5] += (double)bad;
    }
  }
  if (!DIAG) return;
  acc[4] *= 0.5 * rho0;
  __shared__ double red[6][256];
#pragma unroll
  for (int c = 0; c < 6; ++c) red[c][threadIdx.x] = acc[c];
  __syncthreads();
  for (int s = blockDim.x / 2; s > 0; s >>= 1) {
    if ((int)threadIdx.x < s)
#pragma unroll
      for (int c = 0; c < 6; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 6) partial[blockIdx.x * 6 + threadIdx.x] = red[threadIdx.x][0];
}

// one warp per sum: lane partial sums, then a fixed tree (the same order in every run)
__global__ void diag_final_kernel(const double *partial, int nblocks, double *out) {
  const int c = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double s = 0.0;
  for (int b = lane; b < nblocks; b += 32) s += partial[b * 6 + c];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  if (lane == 0) out[c] = s;
}

// fields of unique nodes to local nodes: rho [nloc] (or NULL), u [nloc][dim]
template <int DIM>
__global__ void __launch_bounds__(256) expand_fields_kernel(const double *fld, int G, const int32_t *l2g, size_t nloc,
                                                            double *rho, double *u) {
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < nloc; q += (size_t)gridDim.x * blockDim.x) {
    const size_t g = l2g[q];
    if (rho) rho[q] = fld[g];
#pragma unroll
    for (int k = 0; k < DIM; ++k) u[q * DIM + k] = fld[(size_t)(1 + k) * G + g];
  }
}

template <typename Real, int LAT>
__global__ void __launch_bounds__(256) get_state_kernel(const Real *buf, const int32_t *l2g, int Gs, size_t nloc,
                                                        double rho0, double *f) {
  constexpr VelTab V = LT<LAT>::v;
  constexpr int Q = V.Q, PART = Q == 9 ? 9 : (Q + 2) / 3;
  for (size_t q = blockIdx.x * (size_t)blockDim.x + threadIdx.x; q < nloc; q += (size_t)gridDim.x * blockDim.x) {
    const Real *src = buf + l2g[q];
    static_for<0, (Q + PART - 1) / PART>([&](auto pc) {
      constexpr int a0 = decltype(pc)::value * PART, na = Q - a0 < PART ? Q - a0 : PART;
      Real v[na];
#pragma unroll
      for (int a = 0; a < na; ++a) v[a] = src[(size_t)(a0 + a) * Gs];
      static_for<0, na>([&](auto ac) {
        constexpr int a = decltype(ac)::value;
        f[(size_t)(a0 + a) * nloc + q] = wide(v[a]) + V.t[a0 + a] * rho0;
      });
    });
  }
}

#define SLB_LAT_SWITCH(lat, CALL)                                     \
  switch (lat) {                                                      \
    case SELBM_D2Q9: { constexpr int L = SELBM_D2Q9; CALL; } break;   \
    case SELBM_D3Q19: { constexpr int L = SELBM_D3Q19; CALL; } break; \
    case SELBM_D3Q27: { constexpr int L = SELBM_D3Q27; CALL; } break; \
    default: return cudaErrorInvalidValue;                            \
  }

template <typename Real>
cudaError_t launch_init(int lat, const double *rho, const double *u, const int32_t *first, int G, int Gs, double rho0,
                        double half_dt, const double g[3], int has_force, const Real *fS, double amp, Real *out,
                        cudaStream_t s) {
  SLB_LAT_SWITCH(lat, (init_kernel<Real, L><<<blocks_for(G), 256, 0, s>>>(rho, u, first, G, Gs, rho0, half_dt, g[0], g[1], g[2], has_force, fS, amp, out)));
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_node_fields(int lat, const Real *buf, int G, int Gs, double rho0, double *fld, cudaStream_t s) {
  SLB_LAT_SWITCH(lat, (node_fields_kernel<Real, L, false><<<blocks_for(G), 256, 0, s>>>(buf, G, Gs, rho0, fld, nullptr, nullptr)));
  return cudaGetLastError();
}

int diag_blocks() { return 152 * 4; }
template <typename Real>
cudaError_t launch_diag(int lat, const Real *buf, const double *mass, int G, int Gs, double rho0, double *fld,
                        double *partial, double *out, cudaStream_t s) {
  SLB_LAT_SWITCH(lat, (node_fields_kernel<Real, L, true><<<diag_blocks(), 256, 0, s>>>(buf, G, Gs, rho0, fld, mass, partial)));
  diag_final_kernel<<<1, 6 * 32, 0, s>>>(partial, diag_blocks(), out);
  return cudaGetLastError();
}

cudaError_t launch_expand_fields(int dim, const double *fld, int G, const int32_t *l2g, size_t nloc, double *rho, double *u,
                                 cudaStream_t s) {
  if (dim == 3) expand_fields_kernel<3><<<blocks_for(nloc), 256, 0, s>>>(fld, G, l2g, nloc, rho, u);
  else expand_fields_kernel<2><<<blocks_for(nloc), 256, 0, s>>>(fld, G, l2g, nloc, rho, u);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_get_state(int lat, const Real *buf, const int32_t *l2g, int Gs, size_t nloc, double rho0, double *f,
                             cudaStream_t s) {
  SLB_LAT_SWITCH(lat, (get_state_kernel<Real, L><<<blocks_for(nloc), 256, 0, s>>>(buf, l2g, Gs, nloc, rho0, f)));
  return cudaGetLastError();
}

#define SLB_INST(Real)                                                                                                   \
  template cudaError_t launch_init<Real>(int, const double *, const double *, const int32_t *, int, int, double, double, \
                                         const double[3], int, const Real *, double, Real *, cudaStream_t);              \
  template cudaError_t launch_node_fields<Real>(int, const Real *, int, int, double, double *, cudaStream_t);            \
  template cudaError_t launch_diag<Real>(int, const Real *, const double *, int, int, double, double *, double *,        \
                                         double *, cudaStream_t);                                                        \
  template cudaError_t launch_get_state<Real>(int, const Real *, const int32_t *, int, size_t, double, double *,         \
                                              cudaStream_t);
SLB_INST(float)
SLB_INST(double)

}  // namespace slb
