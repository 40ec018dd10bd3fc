// Instantiations of the any-order element kernels: FP64, orders 2 to 6.
#include "selbm_lines.cuh"

namespace slb {

template <>
cudaError_t lines_stage_part<double, 0>(int N, bool affine, const KParams<double> &p, const SplitHost &h, const LatticeRT &lt,
                                          const LineGeo<double> &lg, cudaStream_t s) {
  switch (N) {
    case 2: return launch_lines_stage_t<double, 3>(affine, p, h, lt, lg, s);
    case 3: return launch_lines_stage_t<double, 4>(affine, p, h, lt, lg, s);
    case 4: return launch_lines_stage_t<double, 5>(affine, p, h, lt, lg, s);
    case 5: return launch_lines_stage_t<double, 6>(affine, p, h, lt, lg, s);
    case 6: return launch_lines_stage_t<double, 7>(affine, p, h, lt, lg, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t lines_filter_part<double, 0>(int N, const KParams<double> &p, const SplitHost &h, int Q, const double *sigma,
                                           double *out, cudaStream_t s) {
  switch (N) {
    case 2: return launch_lines_filter_t<double, 3>(p, h, Q, sigma, out, s);
    case 3: return launch_lines_filter_t<double, 4>(p, h, Q, sigma, out, s);
    case 4: return launch_lines_filter_t<double, 5>(p, h, Q, sigma, out, s);
    case 5: return launch_lines_filter_t<double, 6>(p, h, Q, sigma, out, s);
    case 6: return launch_lines_filter_t<double, 7>(p, h, Q, sigma, out, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
