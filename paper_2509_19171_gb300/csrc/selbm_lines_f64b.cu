// Instantiations of the any-order element kernels: FP64, orders 7 to 9.
#include "selbm_lines.cuh"

namespace slb {

template <>
cudaError_t lines_stage_part<double, 1>(int N, bool affine, const KParams<double> &p, const SplitHost &h, const LatticeRT &lt,
                                          const LineGeo<double> &lg, cudaStream_t s) {
  switch (N) {
    case 7: return launch_lines_stage_t<double, 8>(affine, p, h, lt, lg, s);
    case 8: return launch_lines_stage_t<double, 9>(affine, p, h, lt, lg, s);
    case 9: return launch_lines_stage_t<double, 10>(affine, p, h, lt, lg, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t lines_filter_part<double, 1>(int N, const KParams<double> &p, const SplitHost &h, int Q, const double *sigma,
                                           double *out, cudaStream_t s) {
  switch (N) {
    case 7: return launch_lines_filter_t<double, 8>(p, h, Q, sigma, out, s);
    case 8: return launch_lines_filter_t<double, 9>(p, h, Q, sigma, out, s);
    case 9: return launch_lines_filter_t<double, 10>(p, h, Q, sigma, out, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
