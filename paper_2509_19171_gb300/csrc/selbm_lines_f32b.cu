// Instantiations of the any-order element kernels: FP32, orders 7 to 11.
#include "selbm_lines.cuh"

namespace slb {

template <>
cudaError_t lines_stage_part<float, 1>(int N, bool affine, const KParams<float> &p, const SplitHost &h, const LatticeRT &lt,
                                          const LineGeo<float> &lg, cudaStream_t s) {
  switch (N) {
    case 7: return launch_lines_stage_t<float, 8>(affine, p, h, lt, lg, s);
    case 8: return launch_lines_stage_t<float, 9>(affine, p, h, lt, lg, s);
    case 9: return launch_lines_stage_t<float, 10>(affine, p, h, lt, lg, s);
    case 10: return launch_lines_stage_t<float, 11>(affine, p, h, lt, lg, s);
    case 11: return launch_lines_stage_t<float, 12>(affine, p, h, lt, lg, s);
  }
  return cudaErrorInvalidValue;
}

template <>
cudaError_t lines_filter_part<float, 1>(int N, const KParams<float> &p, const SplitHost &h, int Q, const float *sigma,
                                           float *out, cudaStream_t s) {
  switch (N) {
    case 7: return launch_lines_filter_t<float, 8>(p, h, Q, sigma, out, s);
    case 8: return launch_lines_filter_t<float, 9>(p, h, Q, sigma, out, s);
    case 9: return launch_lines_filter_t<float, 10>(p, h, Q, sigma, out, s);
    case 10: return launch_lines_filter_t<float, 11>(p, h, Q, sigma, out, s);
    case 11: return launch_lines_filter_t<float, 12>(p, h, Q, sigma, out, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
