// Instantiations of the resident 2D step: FP32, orders 2 to 14.
#include "selbm_flow2d.cuh"

namespace slb {

template <>
cudaError_t flow2d_part<float, 0>(int N, bool affine, bool probe, const Flow2DArgs<float> &p, const SplitHost &h,
                                   const Learn2DArgs<float> *lc, bool *fits, cudaStream_t s) {
  switch (N) {
    case 2: return launch_flow2d_t<float, 3, false>(p, h, affine, probe, lc, fits, s);
    case 3: return launch_flow2d_t<float, 4, false>(p, h, affine, probe, lc, fits, s);
    case 4: return launch_flow2d_t<float, 5, false>(p, h, affine, probe, lc, fits, s);
    case 5: return launch_flow2d_t<float, 6, false>(p, h, affine, probe, lc, fits, s);
    case 6: return launch_flow2d_t<float, 7, false>(p, h, affine, probe, lc, fits, s);
    case 7: return launch_flow2d_t<float, 8, false>(p, h, affine, probe, lc, fits, s);
    case 8: return launch_flow2d_t<float, 9, false>(p, h, affine, probe, lc, fits, s);
    case 9: return launch_flow2d_t<float, 10, false>(p, h, affine, probe, lc, fits, s);
    case 10: return launch_flow2d_t<float, 11, false>(p, h, affine, probe, lc, fits, s);
    case 11: return launch_flow2d_t<float, 12, false>(p, h, affine, probe, lc, fits, s);
    case 12: return launch_flow2d_t<float, 13, false>(p, h, affine, probe, lc, fits, s);
    case 13: return launch_flow2d_t<float, 14, false>(p, h, affine, probe, lc, fits, s);
    case 14: return launch_flow2d_t<float, 15, false>(p, h, affine, probe, lc, fits, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
