// Instantiations of the resident 2D step: FP64, orders 2 to 8.
#include "selbm_flow2d.cuh"

namespace slb {

template <>
cudaError_t flow2d_part<double, 0>(int N, bool affine, bool probe, const Flow2DArgs<double> &p, const SplitHost &h,
                                   const Learn2DArgs<double> *lc, bool *fits, cudaStream_t s) {
  switch (N) {
    case 2: return launch_flow2d_t<double, 3, false>(p, h, affine, probe, lc, fits, s);
    case 3: return launch_flow2d_t<double, 4, false>(p, h, affine, probe, lc, fits, s);
    case 4: return launch_flow2d_t<double, 5, false>(p, h, affine, probe, lc, fits, s);
    case 5: return launch_flow2d_t<double, 6, false>(p, h, affine, probe, lc, fits, s);
    case 6: return launch_flow2d_t<double, 7, false>(p, h, affine, probe, lc, fits, s);
    case 7: return launch_flow2d_t<double, 8, false>(p, h, affine, probe, lc, fits, s);
    case 8: return launch_flow2d_t<double, 9, false>(p, h, affine, probe, lc, fits, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
