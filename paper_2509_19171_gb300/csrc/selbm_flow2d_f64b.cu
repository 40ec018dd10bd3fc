// Instantiations of the resident 2D step: FP64, orders 9 to 14.
#include "selbm_flow2d.cuh"

namespace slb {

template <>
cudaError_t flow2d_part<double, 1>(int N, bool affine, bool probe, const Flow2DArgs<double> &p, const SplitHost &h,
                                   const Learn2DArgs<double> *lc, bool *fits, cudaStream_t s) {
  switch (N) {
    case 9: return launch_flow2d_t<double, 10, false>(p, h, affine, probe, lc, fits, s);
    case 10: return launch_flow2d_t<double, 11, false>(p, h, affine, probe, lc, fits, s);
    case 11: return launch_flow2d_t<double, 12, false>(p, h, affine, probe, lc, fits, s);
    case 12: return launch_flow2d_t<double, 13, false>(p, h, affine, probe, lc, fits, s);
    case 13: return launch_flow2d_t<double, 14, false>(p, h, affine, probe, lc, fits, s);
    case 14: return launch_flow2d_t<double, 15, false>(p, h, affine, probe, lc, fits, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
