// Dispatch of the any-order element kernels and of the resident 2D step to the translation units
// of their orders.
#include "selbm_flow2d.cuh"
#include "selbm_lines.cuh"

namespace slb {

template <typename Real>
cudaError_t launch_lines_stage(int lat, int N, bool affine, const KParams<Real> &p, const SplitHost &h,
                               const LineGeo<Real> &lg, cudaStream_t s) {
  const LatticeRT lt = lat == SELBM_D3Q19 ? lattice_rt<SELBM_D3Q19>() : lattice_rt<SELBM_D3Q27>();
  return N <= 6 ? lines_stage_part<Real, 0>(N, affine, p, h, lt, lg, s) : lines_stage_part<Real, 1>(N, affine, p, h, lt, lg, s);
}

template <typename Real>
cudaError_t launch_lines_filter(int lat, int N, const KParams<Real> &p, const SplitHost &h, const Real *sigma, Real *out,
                                cudaStream_t s) {
  const int Q = lat == SELBM_D3Q19 ? LT<SELBM_D3Q19>::v.Q : LT<SELBM_D3Q27>::v.Q;
  return N <= 6 ? lines_filter_part<Real, 0>(N, p, h, Q, sigma, out, s) : lines_filter_part<Real, 1>(N, p, h, Q, sigma, out, s);
}

// affine elements, FP64: -dt sum_k e_k dr_l/dx_k in fixed point, c [E][Q][3] times 2^cexp[E][Q]
__global__ static void affine_geo_kernel(const double *el_drdx, int E, const LatticeRT lt, double dt, long long *c, int *cexp) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= E * lt.Q) return;
  const int e = t / lt.Q, a = t - e * lt.Q;
  double v[3];
  int ex = 1;
  for (int l = 0; l < 3; ++l) {
    double s = 0;
    for (int k = 0; k < 3; ++k)
      s += (double)((int)((lt.pos[k] >> a) & 1u) - (int)((lt.neg[k] >> a) & 1u)) * el_drdx[((size_t)e * 3 + l) * 3 + k];
    v[l] = -dt * s;
    ex = max(ex, exp_of(v[l]));
  }
  cexp[t] = 1082 - ex;                                   // magnitudes below 2^60
  for (int l = 0; l < 3; ++l) c[(size_t)t * 3 + l] = __double2ll_rn(scalbn(v[l], 1082 - ex));
}

cudaError_t launch_affine_geo(int lat, const double *el_drdx, int E, double dt, long long *c, int *cexp, cudaStream_t s) {
  const LatticeRT lt = lat == SELBM_D3Q19 ? lattice_rt<SELBM_D3Q19>() : lattice_rt<SELBM_D3Q27>();
  affine_geo_kernel<<<(E * lt.Q + 255) / 256, 256, 0, s>>>(el_drdx, E, lt, dt, c, cexp);
  return cudaGetLastError();
}

template <typename Real>
cudaError_t launch_flow2d(int N, bool affine, bool probe, const Flow2DArgs<Real> &p, const SplitHost &h, const Learn2DArgs<Real> *lc,
                          bool *fits, cudaStream_t s) {
  if (lc && N < 4) return cudaErrorInvalidValue;
  if (lc) return flow2d_part<Real, 2>(N, affine, probe, p, h, lc, fits, s);
  if constexpr (sizeof(Real) == 8)
    if (N > 8) return flow2d_part<Real, 1>(N, affine, probe, p, h, lc, fits, s);
  return flow2d_part<Real, 0>(N, affine, probe, p, h, lc, fits, s);
}

#define SLB_INST(Real)                                                                                                    \
  template cudaError_t launch_lines_stage<Real>(int, int, bool, const KParams<Real> &, const SplitHost &,                 \
                                                const LineGeo<Real> &, cudaStream_t);                                   \
  template cudaError_t launch_lines_filter<Real>(int, int, const KParams<Real> &, const SplitHost &, const Real *, Real *, \
                                                 cudaStream_t);                                                          \
  template cudaError_t launch_flow2d<Real>(int, bool, bool, const Flow2DArgs<Real> &, const SplitHost &,              \
                                             const Learn2DArgs<Real> *, bool *, cudaStream_t);
SLB_INST(float)
SLB_INST(double)

}  // namespace slb
