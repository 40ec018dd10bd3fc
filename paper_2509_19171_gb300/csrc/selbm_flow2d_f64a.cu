// Instantiations of the resident 2D step: FP64, orders 2 to 8.
#include "selbm_flow2d.cuh"

namespace slb {

template <typename Real, int PART>
cudaError_t flow2d_part(int N, bool affine, bool probe, const Flow2DArgs<Real> &p, const SplitHost &h, bool *fits, cudaStream_t s);

template <>
cudaError_t flow2d_part<double, 0>(int N, bool affine, bool probe, const Flow2DArgs<double> &p, const SplitHost &h, bool *fits,
                                   cudaStream_t s) {
  switch (N) {
    case 2: return launch_flow2d_t<double, 3>(p, h, affine, probe, fits, s);
    case 3: return launch_flow2d_t<double, 4>(p, h, affine, probe, fits, s);
    case 4: return launch_flow2d_t<double, 5>(p, h, affine, probe, fits, s);
    case 5: return launch_flow2d_t<double, 6>(p, h, affine, probe, fits, s);
    case 6: return launch_flow2d_t<double, 7>(p, h, affine, probe, fits, s);
    case 7: return launch_flow2d_t<double, 8>(p, h, affine, probe, fits, s);
    case 8: return launch_flow2d_t<double, 9>(p, h, affine, probe, fits, s);
  }
  return cudaErrorInvalidValue;
}

}  // namespace slb
