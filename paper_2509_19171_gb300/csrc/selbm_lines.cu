// Dispatch of the any-order element kernels and of the resident 2D step to the translation units
// of their orders.
#include "selbm_flow2d.cuh"
#include "selbm_lines.cuh"

namespace slb {

template <typename Real>
cudaError_t launch_lines_stage(int lat, int N, bool affine, const KParams<Real> &p, const SplitHost &h,
                               const CurvedGeo<Real> &cg, cudaStream_t s) {
  const LatticeRT lt = lat == SELBM_D3Q19 ? lattice_rt<SELBM_D3Q19>() : lattice_rt<SELBM_D3Q27>();
  return N <= 6 ? lines_stage_part<Real, 0>(N, affine, p, h, lt, cg, s) : lines_stage_part<Real, 1>(N, affine, p, h, lt, cg, s);
}

template <typename Real>
cudaError_t launch_lines_filter(int lat, int N, const KParams<Real> &p, const SplitHost &h, const Real *sigma, Real *out,
                                cudaStream_t s) {
  const int Q = lat == SELBM_D3Q19 ? LT<SELBM_D3Q19>::v.Q : LT<SELBM_D3Q27>::v.Q;
  return N <= 6 ? lines_filter_part<Real, 0>(N, p, h, Q, sigma, out, s) : lines_filter_part<Real, 1>(N, p, h, Q, sigma, out, s);
}

template <typename Real>
cudaError_t launch_curved_geo(const Real *drdx, int E, int Np, LineVal<Real> *g, int *gexp, cudaStream_t s) {
  curved_geo_kernel<Real><<<E, 256, 0, s>>>(drdx, Np, g, gexp);
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
                                                const CurvedGeo<Real> &, cudaStream_t);                                   \
  template cudaError_t launch_lines_filter<Real>(int, int, const KParams<Real> &, const SplitHost &, const Real *, Real *, \
                                                 cudaStream_t);                                                          \
  template cudaError_t launch_curved_geo<Real>(const Real *, int, int, LineVal<Real> *, int *, cudaStream_t);             \
  template cudaError_t launch_flow2d<Real>(int, bool, bool, const Flow2DArgs<Real> &, const SplitHost &,              \
                                             const Learn2DArgs<Real> *, bool *, cudaStream_t);
SLB_INST(float)
SLB_INST(double)

}  // namespace slb
