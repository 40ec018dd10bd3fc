// Instantiations of the any-order element kernels: FP32, orders 2 to 6.
#include "selbm_lines.cuh"

namespace slb {

template <>
cudaError_t lines_stage_part<float, 0>(int N, bool affine, const KParams<float> &p, const SplitHost &h, const LatticeRT &lt,
                                          const LineGeo<float> &lg, cudaStream_t s) {
  switch (N) {
    case 2: return launch_lines_stage_t<float, 3>(affine, p, h, lt, lg, s);
    case 3: return launch_lines_stage_t<float, 4>(affine, p, h, lt, lg, s);
    case 4: return launch_lines_stage_t<float, 5>(affine, p, h, lt, lg, s);
    case 5: return launch_lines_stage_t<float, 6>(affine, p, h, lt, lg, s);
    case 6: return launch_lines_stage_t<float, 7>(affine, p, h, lt, lg, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t lines_filter_part<float, 0>(int N, const KParams<float> &p, const SplitHost &h, int Q, const float *sigma,
                                           float *out, cudaStream_t s) {
  switch (N) {
    case 2: return launch_lines_filter_t<float, 3>(p, h, Q, sigma, out, s);
    case 3: return launch_lines_filter_t<float, 4>(p, h, Q, sigma, out, s);
    case 4: return launch_lines_filter_t<float, 5>(p, h, Q, sigma, out, s);
    case 5: return launch_lines_filter_t<float, 6>(p, h, Q, sigma, out, s);
    case 6: return launch_lines_filter_t<float, 7>(p, h, Q, sigma, out, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
