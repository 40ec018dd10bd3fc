// Any-order element kernels of the population-split step (hexahedra): host interface.
#pragma once
#include <type_traits>

#include "selbm_fixed_lines.cuh"
#include "selbm_kernels.cuh"

namespace slb {

// velocity set at run time
struct LatticeRT {
  int Q;
  uint32_t pos[3], neg[3];
  float tf[27];
  double td[27];
  signed char opp[27];
  template <typename Real>
  __device__ __forceinline__ Real t(int a) const {
    if constexpr (sizeof(Real) == 8) return td[a];
    else return tf[a];
  }
};

// tables of the stage kernel beside the metrics.  Affine elements, FP64: -dt sum_k e_k dr_l/dx_k [E][Q][3] in fixed
// point, times 2^gexp[e Q + a], and the quadrature weights w w w [Np].  Curved elements, FP64: gexp[e], the
// largest biased exponent of the element's metrics.
template <typename Real>
struct LineGeo {
  const LineVal<Real> *g;
  const int *gexp;
  const Real *w3;
};

// orders whose element tile fits the step's other kernels too (real_size 4 or 8)
inline bool lines_compiled(int real_size, int N) { return N >= 2 && N <= (real_size == 8 ? 9 : 11); }

// one Runge-Kutta stage of the element kernels (see selbm_split_stage.cuh for its terms)
template <typename Real>
cudaError_t launch_lines_stage(int lat, int N, bool affine, const KParams<Real> &p, const SplitHost &h,
                               const LineGeo<Real> &lg, cudaStream_t s);
// filtered p.fin: sigma NULL: the fixed filter, every unique node to out; else element transfer
// functions sigma [E][n], element-interior nodes to out and shares wJ f of the others to p.T
template <typename Real>
cudaError_t launch_lines_filter(int lat, int N, const KParams<Real> &p, const SplitHost &h, const Real *sigma, Real *out,
                                cudaStream_t s);
// the affine FP64 tables from el_drdx [E][3][3]
cudaError_t launch_affine_geo(int lat, const double *el_drdx, int E, double dt, long long *c, int *cexp, cudaStream_t s);

}  // namespace slb
