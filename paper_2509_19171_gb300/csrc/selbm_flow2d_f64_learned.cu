// Instantiations of the resident 2D step: FP64, orders 4 to 14, with the learned control.
#include "selbm_flow2d.cuh"

namespace slb {

template <>
cudaError_t flow2d_part<double, 2>(int N, bool affine, bool probe, const Flow2DArgs<double> &p, const SplitHost &h,
                                   const Learn2DArgs<double> *lc, bool *fits, cudaStream_t s) {
  switch (N) {
    case 4: return launch_flow2d_t<double, 5, true>(p, h, affine, probe, lc, fits, s);
    case 5: return launch_flow2d_t<double, 6, true>(p, h, affine, probe, lc, fits, s);
    case 6: return launch_flow2d_t<double, 7, true>(p, h, affine, probe, lc, fits, s);
    case 7: return launch_flow2d_t<double, 8, true>(p, h, affine, probe, lc, fits, s);
    case 8: return launch_flow2d_t<double, 9, true>(p, h, affine, probe, lc, fits, s);
    case 9: return launch_flow2d_t<double, 10, true>(p, h, affine, probe, lc, fits, s);
    case 10: return launch_flow2d_t<double, 11, true>(p, h, affine, probe, lc, fits, s);
    case 11: return launch_flow2d_t<double, 12, true>(p, h, affine, probe, lc, fits, s);
    case 12: return launch_flow2d_t<double, 13, true>(p, h, affine, probe, lc, fits, s);
    case 13: return launch_flow2d_t<double, 14, true>(p, h, affine, probe, lc, fits, s);
    case 14: return launch_flow2d_t<double, 15, true>(p, h, affine, probe, lc, fits, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
